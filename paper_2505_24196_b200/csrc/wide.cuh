// Layers over many rows (a prompt fed in large pieces, wide candidate sets): the products are
// bound by the tensor cores, not by the weight stream, so the work split differs from the
// skinny kernels: activation rows sit on the MMA's M axis, 256 features on its N axis.
//
//   gemm_kernel   y = x W^T, one CTA pair per 256 x 256 tile (tcgen05 cta_group::2), persistent
//   attn_kernel   causal attention over cache and own rows, 128 (row, query head) pairs per CTA
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gemm_tc.cuh"
#include "kernels.cuh"

namespace clasp {
namespace wide {

using bf16 = __nv_bfloat16;

constexpr int BK = 64;            // one 128-byte swizzle row of bf16
constexpr int TM = 128;           // activation rows per CTA (tensor-memory lanes)
constexpr int TN = 256;           // features per tile; each CTA of the pair loads 128 of them
constexpr int STAGES = 6;
constexpr int STAGE_BYTES = (TM + TN / 2) * BK * 2;   // 32 KB per CTA
constexpr int GEMM_THREADS = 384; // warp 0 TMA, warp 1 MMA, warp 2 tensor memory, warps 4-11 epilogue
constexpr int GEMM_SMEM = STAGES * STAGE_BYTES + 1024;
constexpr int SLOT_FLOATS = TM * TN;                  // one CTA's share of a tile, as partial sums

struct GemmParams {
  int R, kc;               // rows, 64-column chunks of K
  int n_mats;              // 1..3 matrices stacked along the features
  int N[3], f_tiles[3], col_off[3];
  int row_tiles, tiles;    // 256-row tiles; all tiles
  int sk_tiles, sk_pairs;  // tiles [0, sk_tiles) are split over K among the first sk_pairs pairs, the others go to one pair each
  int dual, epi;
  float* yf;
  long long ldy;
  const float* resid;
  long long ldr;
  bf16* yo;
  long long ldo;
  float* partial;          // [CTA][2][SLOT_FLOATS]
  int* counters;           // [sk_tiles][2], zero on entry and on exit
  int* status;
  uint32_t spin_fast, spin_slow;
};

__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred;
}
// the same place in the shared memory of the pair's even CTA
__device__ __forceinline__ uint32_t leader_addr(uint32_t a) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(a));
  return r;
}
// a load into this CTA's shared memory that reports its bytes to a barrier of the even CTA (leader_addr)
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;"
      :
      : "r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, bool acc, uint32_t el) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "setp.ne.u32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(da), "l"(db), "r"(idesc), "r"((uint32_t)acc), "r"(el)
      : "memory");
}
// arrives on the barrier at this address in both CTAs once the MMAs issued so far are done
__device__ __forceinline__ void commit_pair(uint32_t bar, uint32_t el) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %2;\n\t}" ::"r"(bar),
      "r"(el), "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void arrive_leader(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(leader_addr(bar)) : "memory");
}
// eight floats (32 bytes): one access where the address allows it.  Predicated inside the statement: the warp stays
// converged for the tensor-memory reads around it.
__device__ __forceinline__ void st8(float* p, const float* v, bool al32, bool on) {
  if (al32) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %9, 0;\n\t@q st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n\t}"
                 ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "r"((uint32_t)on)
                 : "memory");
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %5, 0;\n\t@q st.global.v4.f32 [%0], {%1, %2, %3, %4};\n\t}"
                   ::"l"(p + 4 * h), "f"(v[4 * h]), "f"(v[4 * h + 1]), "f"(v[4 * h + 2]), "f"(v[4 * h + 3]), "r"((uint32_t)on)
                   : "memory");
  }
}
__device__ __forceinline__ void st16b(void* p, uint32_t a, uint32_t b, uint32_t c, uint32_t d, bool on) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %5, 0;\n\t@q st.global.v4.b32 [%0], {%1, %2, %3, %4};\n\t}"
               ::"l"(p), "r"(a), "r"(b), "r"(c), "r"(d), "r"((uint32_t)on)
               : "memory");
}
__device__ __forceinline__ void ld8(const float* p, float* v, bool al32) {
  if (al32) {
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p));
  } else {
    const float4 a = __ldcg(reinterpret_cast<const float4*>(p)), b = __ldcg(reinterpret_cast<const float4*>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
}
__device__ __forceinline__ uint32_t pack2(float x, float y) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<const uint32_t*>(&h);
}
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[N]) {
  static_assert(N == 8 || N == 32, "accumulator columns per read");
  uint32_t r[N];
  if constexpr (N == 8) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
  } else {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
  }
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

// ------------------------------------------------------------------ the products
// Work list of a pair w of W: first its share of the tiles that are split over K -- all their (tile, chunk) units in one
// row, cut into sk_pairs equal ranges --, then whole tiles w, w + W, ...  The split part, if any, is what whole waves of tiles
// leave over.
struct Items {
  long long u, u1;
  int dp, W;
  __device__ __forceinline__ static long long start(const GemmParams& p, int w) {
    return (long long)p.sk_tiles * p.kc * min(w, p.sk_pairs) / p.sk_pairs;
  }
  __device__ __forceinline__ Items(const GemmParams& p, int w, int W_) : W(W_) {
    u = start(p, w);
    u1 = start(p, w + 1);
    dp = p.sk_tiles + w;
  }
  __device__ __forceinline__ bool next(const GemmParams& p, int& tile, int& kb, int& ke) {
    if (u < u1) {
      tile = (int)(u / p.kc);
      kb = (int)(u - (long long)tile * p.kc);
      ke = (int)min((long long)p.kc, kb + (u1 - u));
      u += ke - kb;
      return true;
    }
    if (dp < p.tiles) {
      tile = dp;
      kb = 0;
      ke = p.kc;
      dp += W;
      return true;
    }
    return false;
  }
};

// Row tiles are the inner index of the tile order: the pairs at work at one time share few weight tiles.
struct TileAt {
  int mat, f0, m0;   // matrix, first feature in it, first row
  __device__ __forceinline__ TileAt(const GemmParams& p, int tile) {
    int ft = tile / p.row_tiles;
    m0 = (tile - ft * p.row_tiles) * (2 * TM);
    mat = 0;
    while (mat + 1 < p.n_mats && ft >= p.f_tiles[mat]) { ft -= p.f_tiles[mat]; ++mat; }
    f0 = ft * (p.dual ? TN / 2 : TN);
  }
};

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
// Barrier of the eight epilogue warps that also tells whether p holds in any of them.  After a wait each warp polls for itself,
// and the polls of one may run out just before another's succeed: they go on, or leave, together -- a warp that left alone
// would be missing at the barriers of the others, which have no limit.
__device__ __forceinline__ bool epi_any(bool p) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred a, b;\n\tsetp.ne.u32 a, %1, 0;\n\tbar.red.or.pred b, 1, 256, a;\n\tselp.u32 %0, 1, 0, b;\n\t}"
               : "=r"(r)
               : "r"((uint32_t)p)
               : "memory");
  return r != 0;
}

// y[r, n] = sum_k x[r, k] w[n, k] over tiles of 256 rows x 256 features (SwiGLU: 128 gate and 128 up features).  A pair
// of CTAs multiplies a tile: each loads 128 rows of x and 128 rows of W, the even CTA issues M = 256 MMAs that read
// both, each keeps the accumulator of its own 128 rows.  A 64-column chunk is 512 cycles of multiplies for 32 KB of loads
// per SM (one CTA per tile of 128 x 256 would need 48 KB for the same work).  Measured, 8B shape, 1999 rows, PFLOP/s in a
// loop under the power cap, a plain library product of the same shape beside it: gate/up 1.22 / 1.25, q/k/v 1.06 / 1.27, o
// 0.94 / 1.28, down 1.11 / 1.32.  Gate/up is at the power cap.  The others have two or three waves of tiles (o and down 1.7 of
// 2, q/k/v 2.6 of 3); their loads, 64 KB per pair and chunk, come to 11.6 TB/s for gate/up and 9.0, 7.9 and 9.7 for q/k/v, o
// and down, so the rate of L2 does not bound them, and what takes the rest is not known.  (Passes of 256 rows through the
// skinny product, which re-read all weights eight times, and the CUDA-core attention took 14.9 ms per layer together.)  At
// 128 rows the four products take 216 us against 114 inside the persistent kernel (partial sums, ramps), so that kernel
// keeps the launches of up to 128 rows.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GEMM_THREADS, 1)
gemm_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w0,
            const __grid_constant__ CUtensorMap map_w1, const __grid_constant__ CUtensorMap map_w2, const GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_full[STAGES], bar_empty[STAGES], acc_full[2], acc_empty[2];
  __shared__ uint32_t s_tmem_base;
  __shared__ int s_abort, s_is_last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank();
  const int w = blockIdx.x >> 1, W = gridDim.x >> 1;
  const uint32_t ring = (tc::smem_u32(smem_raw) + 1023u) & ~1023u;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      tc::mbar_init(tc::smem_u32(&bar_full[s]), 1);
      tc::mbar_init(tc::smem_u32(&bar_empty[s]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(tc::smem_u32(&acc_full[b]), 1);
      tc::mbar_init(tc::smem_u32(&acc_empty[b]), 2);   // the epilogues of both CTAs
    }
    s_abort = 0;
    s_is_last = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&s_tmem_base)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync();   // the peer's barriers exist
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = s_tmem_base;

  if (warp == 0) {
    if (lane == 0) {
      uint64_t pol;
      asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
      Items items(p, w, W);
      int tile, kb, ke;
      uint32_t n = 0;
      bool ok = true;
      while (ok && items.next(p, tile, kb, ke)) {
        const TileAt t(p, tile);
        // feature rows of this CTA: its half of the tile, or (SwiGLU) the tile's rows of "its" matrix
        const CUtensorMap* mw = p.dual ? (rank ? &map_w1 : &map_w0) : (t.mat == 0 ? &map_w0 : (t.mat == 1 ? &map_w1 : &map_w2));
        const int wy = t.f0 + (p.dual ? 0 : (int)rank * (TN / 2));
        const int xy = t.m0 + (int)rank * TM;
        for (int k = kb; k < ke; ++k, ++n) {
          const uint32_t s = n % STAGES;
          if (!tc::mbar_wait(tc::smem_u32(&bar_empty[s]), ((n / STAGES) & 1u) ^ 1u, p.status, p.spin_fast, p.spin_slow)) { ok = false; break; }
          const uint32_t full = tc::smem_u32(&bar_full[s]);
          const uint32_t dst = ring + s * STAGE_BYTES, full0 = leader_addr(full);
          if (rank == 0) tc::mbar_expect_tx(full, 2 * STAGE_BYTES);
          tma_load_pair(dst, &map_x, full0, k * BK, xy, pol);
          tma_load_pair(dst + TM * BK * 2, mw, full0, k * BK, wy, pol);
        }
      }
      if (!ok) s_abort = 1;
    }
  } else if (warp == 1) {
    if (rank == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(2 * TM >> 4) << 24);
      const uint32_t el = elect_one();
      Items items(p, w, W);
      int tile, kb, ke;
      uint32_t n = 0, n_acc = 0;
      bool ok = true;
      while (ok && items.next(p, tile, kb, ke)) {
        const uint32_t buf = n_acc & 1u;
        ok = tc::mbar_wait(tc::smem_u32(&acc_empty[buf]), ((n_acc >> 1) & 1u) ^ 1u, p.status, p.spin_fast, p.spin_slow);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc = tmem_base + buf * TN;
        for (int k = kb; k < ke; ++k, ++n) {
          const uint32_t s = n % STAGES;
          ok = tc::mbar_wait(tc::smem_u32(&bar_full[s]), (n / STAGES) & 1u, p.status, p.spin_fast, p.spin_slow);
          if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t da = tc::make_smem_desc(ring + s * STAGE_BYTES);
          const uint64_t db = tc::make_smem_desc(ring + s * STAGE_BYTES + TM * BK * 2);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) mma_pair(acc, da + 2 * kk, db + 2 * kk, idesc, k > kb || kk > 0, el);
          commit_pair(tc::smem_u32(&bar_empty[s]), el);
        }
        if (!ok) break;
        commit_pair(tc::smem_u32(&acc_full[buf]), el);
        ++n_acc;
      }
      if (!ok) s_abort = 1;
    }
  } else if (warp >= 4) {
    // epilogue: thread (quarter, lane) owns a row, warps w and w + 4 take one half of the columns each
    const int ew = warp - 4, quarter = ew & 3, half = ew >> 2, etid = (int)threadIdx.x - 128;
    const int row_l = quarter * 32 + lane;
    Items items(p, w, W);
    int tile, kb, ke;
    uint32_t n_acc = 0;
    const bool al_y = ((uintptr_t)p.yf & 31) == 0 && (p.ldy & 7) == 0;
    const bool al_r = ((uintptr_t)p.resid & 31) == 0 && (p.ldr & 7) == 0;
    while (items.next(p, tile, kb, ke)) {
      const TileAt t(p, tile);
      const uint32_t buf = n_acc & 1u;
      const bool ok = tc::mbar_wait(tc::smem_u32(&acc_full[buf]), (n_acc >> 1) & 1u, p.status, p.spin_fast, p.spin_slow);
      __syncwarp();
      if (epi_any(!ok)) { s_abort = 1; break; }   // (a part of a split tile is then never counted: the status call clears the counters)
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t t_row = tmem_base + buf * TN + ((uint32_t)(quarter * 32) << 16);
      const int r = t.m0 + (int)rank * TM + row_l;
      const bool rv = r < p.R;
      int first = 0, last = 0;     // pairs that hold parts of this tile
      bool finish = true;
      if (kb > 0 || ke < p.kc) {
        // a part of the tile: partial sums to the workspace; the pair that comes last adds all parts in pair order
        const long long t0 = (long long)tile * p.kc, t1 = t0 + p.kc;
        const long long U = (long long)p.sk_tiles * p.kc;
        first = (int)(t0 * p.sk_pairs / U);
        while (Items::start(p, first + 1) <= t0) ++first;
        while (Items::start(p, first) > t0) --first;
        last = first;
        while (Items::start(p, last + 1) < t1) ++last;
        float* slot = p.partial + ((long long)blockIdx.x * 2 + (Items::start(p, w) >= t0 ? 0 : 1)) * SLOT_FLOATS;
#pragma unroll 1
        for (int c = half * (TN / 2); c < (half + 1) * (TN / 2); c += 32) {
          float v[32];
          tmem_ld<32>(t_row + c, v);
          tmem_wait_ld();
#pragma unroll
          for (int g = 0; g < 4; ++g) st8(slot + ((long long)(c / 8 + g) * TM + row_l) * 8, v + 8 * g, true, true);
        }
        __threadfence();
        epi_sync();
        if (etid == 0) {
          int* cnt = p.counters + tile * 2 + rank;
          s_is_last = atomicAdd(cnt, 1) == last - first;
          if (s_is_last) *cnt = 0;
        }
        epi_sync();
        finish = s_is_last != 0;
        if (finish) __threadfence();
      }
      // N columns of the finished tile, from tensor memory or as the sum of the parts
      auto columns = [&](int c, auto& v) {
        constexpr int NC = sizeof(v) / sizeof(float);
        if (last == first) {
          tmem_ld<NC>(t_row + c, v);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int i = 0; i < NC; ++i) v[i] = 0.f;
          const long long t0 = (long long)tile * p.kc;
          for (int ww = first; ww <= last; ++ww) {
            const float* slot = p.partial + ((long long)(ww * 2 + (int)rank) * 2 + (Items::start(p, ww) >= t0 ? 0 : 1)) * SLOT_FLOATS;
#pragma unroll
            for (int g = 0; g < NC / 8; ++g) {
              const float4* q = reinterpret_cast<const float4*>(slot + ((long long)(c / 8 + g) * TM + row_l) * 8);
              const float4 a = __ldcg(q), b = __ldcg(q + 1);
              float* d = v + 8 * g;
              d[0] += a.x; d[1] += a.y; d[2] += a.z; d[3] += a.w; d[4] += b.x; d[5] += b.y; d[6] += b.z; d[7] += b.w;
            }
          }
        }
      };
      if (finish) {
        const int n_f = p.N[t.mat];
        const long long rr = min(r, p.R - 1);   // (rows past the end: loads stay inside, stores are off)
        if (p.epi == EPI_SWIGLU) {
#pragma unroll 1
          for (int c = half * (TN / 4); c < (half + 1) * (TN / 4); c += 32) {
            float g[32], u[32];
            columns(c, g);
            columns(TN / 2 + c, u);
            bf16* dst = p.yo + rr * p.ldo + t.f0 + c;   // 16-byte aligned: widths are multiples of 8
#pragma unroll
            for (int h = 0; h < 4; ++h) {
              uint32_t o[4];
#pragma unroll
              for (int i = 0; i < 4; ++i)
                o[i] = pack2(tc::silu(g[8 * h + 2 * i]) * u[8 * h + 2 * i], tc::silu(g[8 * h + 2 * i + 1]) * u[8 * h + 2 * i + 1]);
              st16b(dst + 8 * h, o[0], o[1], o[2], o[3], rv && t.f0 + c + 8 * h < n_f);
            }
          }
        } else {
          const bool res = p.epi == EPI_RESID;
          const long long col = p.col_off[t.mat] + t.f0;
#pragma unroll 1
          for (int c = half * (TN / 2); c < (half + 1) * (TN / 2); c += 32) {
            float v[32], x[32];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
#pragma unroll
              for (int i = 0; i < 8; ++i) x[8 * g + i] = 0.f;
              if (res && t.f0 + c + 8 * g < n_f) ld8(p.resid + rr * p.ldr + col + c + 8 * g, x + 8 * g, al_r);
            }
            columns(c, v);
            if (res) {
#pragma unroll
              for (int i = 0; i < 32; ++i) v[i] = x[i] + v[i];
            }
#pragma unroll
            for (int g = 0; g < 4; ++g)
              st8(p.yf + rr * p.ldy + col + c + 8 * g, v + 8 * g, al_y, rv && t.f0 + c + 8 * g < n_f);
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      epi_sync();
      if (etid == 0) arrive_leader(tc::smem_u32(&acc_empty[buf]));
      ++n_acc;
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (s_abort) {
    // a wait gave up: copies and MMAs still in flight land before shared and tensor memory are released
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
  cluster_sync();   // nothing of the peer still writes here
  if (warp == 2) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

// ------------------------------------------------------------------ attention
constexpr int HD = 128;
constexpr int ATT_PAIRS = 128;    // (row, query head) pairs of one kv head per CTA: tensor-memory lanes
constexpr int ATT_TK = 64;        // keys per tile
constexpr int ATT_RING = 3;       // K and V tiles in flight
constexpr int ATT_THREADS = 192;  // warps 0-3 softmax (a thread per pair), warp 4 TMA, warp 5 MMA
constexpr uint32_t Q_BYTES = ATT_PAIRS * HD * 2;
constexpr uint32_t KV_BYTES = ATT_TK * HD * 2;
constexpr int ATT_SMEM = 2 * Q_BYTES + ATT_RING * KV_BYTES + 256;   // two CTAs per SM
// tensor-memory columns: two score buffers (their weights overwrite them, high and low halves of 32 columns), the output
constexpr uint32_t S_COL = 0, O_COL = 128;

struct AttnParams {
  const float* qkv;
  long long ldq;
  const float2* cs;
  int C, R, T, nq, nkv;
  int blocks;              // blocks of ATT_PAIRS pairs per kv head
  int splits;              // parts of each block's key tiles
  bf16* out;               // splits == 1: [R, nq * HD]
  float* part_acc;         // else: [R * nq, splits, HD] and
  float2* part_ml;         //       [R * nq, splits] (maximum, sum) for attn_merge_kernel
  int* status;
  uint32_t spin_fast, spin_slow;
};

struct AttnShared {
  uint64_t kv_full[ATT_RING], kv_empty[ATT_RING], s_full[2], p_full[2];
  uint64_t o_done[2];   // by parity of the tile: a wait that skips tiles may lag one behind, never two
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(AttnShared) <= 256, "barriers fit their share of shared memory");

// accumulate: D = A B + D with A (bf16 pairs, one row per lane) in tensor memory
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t db, uint32_t idesc, bool acc, uint32_t el) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "setp.ne.u32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
      "r"(a), "l"(db), "r"(idesc), "r"((uint32_t)acc), "r"(el)
      : "memory");
}
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t da, uint64_t db, uint32_t idesc, bool acc, uint32_t el) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %4, 0;\n\t"
      "setp.ne.u32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(da), "l"(db), "r"(idesc), "r"((uint32_t)acc), "r"(el)
      : "memory");
}
__device__ __forceinline__ void commit_one(uint32_t bar, uint32_t el) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar), "r"(el)
      : "memory");
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// x = hi + lo with both bf16: 16 bits of x's mantissa
__device__ __forceinline__ void split2(float x, float y, uint32_t& hi, uint32_t& lo) {
  hi = pack2(x, y);
  lo = pack2(x - __uint_as_float(hi << 16), y - __uint_as_float(hi & 0xffff0000u));
}

// Attention of the rows' queries over the cache keys [0, C) and the own rows (row r sees own rows of its state, of T
// rows, up to itself).  A CTA takes ATT_PAIRS pairs (row, query head) of one kv head through its key tiles:
//   S = Q K^T, softmax weights P = exp2(S - m), O += P V, all multiplies on tcgen05, S / P / O in tensor memory.
// Queries and weights enter their product as a bf16 pair each (high + low part, two multiplies): 17 bits where the attention
// on the CUDA cores held 24.  What that leaves is far below the rounding of the result to the bf16 operand of the o
// projection: error of the attention alone against float64, weights that cancel, 1.6457e-3 - 1.6621e-3 with fp32 operands'
// 1.6454e-3 - 1.6619e-3 beside it, of 52 prompts of 129 - 1000 rows 0.9999 +- 0.0002 times as large.  A thread owns a pair; its maximum m moves only when exceeded by more than 2^8 (then O is rescaled).
// Scores are double-buffered so that the next tile's Q K^T runs under this tile's softmax, and two CTAs share an SM.
// Bound by the multiplies (four per score and value because of the two parts): 84 us per layer at 1999 rows, 32 query
// heads, where the tensor pipe alone needs about 30.
__global__ void __launch_bounds__(ATT_THREADS, 2)
attn_kernel(const __grid_constant__ CUtensorMap map_ck, const __grid_constant__ CUtensorMap map_cv,
            const __grid_constant__ CUtensorMap map_ok, const __grid_constant__ CUtensorMap map_ov, const AttnParams p) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t base = tc::smem_u32(smem);
  AttnShared* sh = reinterpret_cast<AttnShared*>(smem + 2 * Q_BYTES + ATT_RING * KV_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Gq = p.nq / p.nkv, Pn = p.R * Gq;
  // longest blocks first
  int b = blockIdx.x;
  const int split = b % p.splits;
  b /= p.splits;
  const int kvh = b % p.nkv;
  const int blk = p.blocks - 1 - b / p.nkv;
  const int pair0 = blk * ATT_PAIRS;
  const int r_lo = pair0 / Gq, r_hi = min(p.R - 1, (pair0 + ATT_PAIRS - 1) / Gq);
  const int own_lo = r_lo / p.T * p.T;                                   // first own key any of the rows sees
  const int nt_c = (p.C + ATT_TK - 1) / ATT_TK, nt_all = nt_c + (r_hi - own_lo) / ATT_TK + 1;
  const int t_lo = (int)((long long)nt_all * split / p.splits), nt = (int)((long long)nt_all * (split + 1) / p.splits) - t_lo;

  if ((base & 1023u) != 0) {   // the tiles' swizzle needs it (dynamic shared memory starts aligned)
    if (threadIdx.x == 0) atomicExch(p.status, 1);
    return;
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < ATT_RING; ++s) {
      tc::mbar_init(tc::smem_u32(&sh->kv_full[s]), 1);
      tc::mbar_init(tc::smem_u32(&sh->kv_empty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(tc::smem_u32(&sh->s_full[s]), 1);
      tc::mbar_init(tc::smem_u32(&sh->p_full[s]), ATT_PAIRS);
      tc::mbar_init(tc::smem_u32(&sh->o_done[s]), 1);
    }
    sh->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 5) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&sh->tmem_base)), "r"(256u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (warp < 4) {
    // query rows, rotated and scaled, as two bf16 parts: dims i and i + 64 of a row share a rotation, so a thread makes
    // the pieces (row, j) and (row, j + 8) from the same loads
    const float qscale = rsqrtf((float)HD) * 1.4426950408889634f;
#pragma unroll 2
    for (int e = 0; e < ATT_PAIRS * 8 / 128; ++e) {
      const int task = (int)threadIdx.x + e * 128;
      const int qrow = task >> 3, j = task & 7;
      const int pp = pair0 + qrow;
      uint32_t h0[4] = {0, 0, 0, 0}, l0[4] = {0, 0, 0, 0}, h1[4] = {0, 0, 0, 0}, l1[4] = {0, 0, 0, 0};
      if (pp < Pn) {
        const int rr = pp / Gq, hq = kvh * Gq + pp % Gq;
        const float* qr = p.qkv + (long long)rr * p.ldq + hq * HD + j * 8;
        const float4 a0 = *reinterpret_cast<const float4*>(qr), a1 = *reinterpret_cast<const float4*>(qr + 4);
        const float4 b0 = *reinterpret_cast<const float4*>(qr + HD / 2), b1 = *reinterpret_cast<const float4*>(qr + HD / 2 + 4);
        const float4* cs4 = reinterpret_cast<const float4*>(p.cs + (long long)(rr % p.T) * (HD / 2) + j * 8);
        const float lo[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
        const float hi[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 cs = cs4[q];
          split2((lo[2 * q] * cs.x - hi[2 * q] * cs.y) * qscale, (lo[2 * q + 1] * cs.z - hi[2 * q + 1] * cs.w) * qscale, h0[q], l0[q]);
          split2((hi[2 * q] * cs.x + lo[2 * q] * cs.y) * qscale, (hi[2 * q + 1] * cs.z + lo[2 * q + 1] * cs.w) * qscale, h1[q], l1[q]);
        }
      }
      uint8_t* dst = smem + qrow * 128 + ((j ^ (qrow & 7)) << 4);
      *reinterpret_cast<uint4*>(dst) = make_uint4(h0[0], h0[1], h0[2], h0[3]);
      *reinterpret_cast<uint4*>(dst + ATT_PAIRS * 128) = make_uint4(h1[0], h1[1], h1[2], h1[3]);
      *reinterpret_cast<uint4*>(dst + Q_BYTES) = make_uint4(l0[0], l0[1], l0[2], l0[3]);
      *reinterpret_cast<uint4*>(dst + Q_BYTES + ATT_PAIRS * 128) = make_uint4(l1[0], l1[1], l1[2], l1[3]);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sh->tmem_base;

  if (warp == 4) {
    if (lane == 0) {
      // tiles in the order the multiplies take them: K0, K1, V0, K2, V1, ...
      uint64_t pol;
      asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
      uint32_t n = 0;
      bool ok = true;
      auto load = [&](bool value, int t) {
        const uint32_t s = n % ATT_RING;
        ok = tc::mbar_wait(tc::smem_u32(&sh->kv_empty[s]), ((n / ATT_RING) & 1u) ^ 1u, p.status, p.spin_fast, p.spin_slow);
        if (!ok) return;
        const int tt = t_lo + t;
        const bool own = tt >= nt_c;
        const CUtensorMap* m = own ? (value ? &map_ov : &map_ok) : (value ? &map_cv : &map_ck);
        const int y = own ? own_lo + (tt - nt_c) * ATT_TK : tt * ATT_TK;
        const uint32_t bar = tc::smem_u32(&sh->kv_full[s]), dst = base + 2 * Q_BYTES + s * KV_BYTES;
        tc::mbar_expect_tx(bar, KV_BYTES);
        tc::tma_load_2d(dst, m, bar, kvh * HD, y, pol);
        tc::tma_load_2d(dst + KV_BYTES / 2, m, bar, kvh * HD + HD / 2, y, pol);
        ++n;
      };
      if (nt > 0) load(false, 0);
      for (int t = 0; t < nt && ok; ++t) {
        if (t + 1 < nt) load(false, t + 1);
        if (ok) load(true, t);
      }
      if (!ok) sh->abort = 1;
    }
  } else if (warp == 5) {
    const uint32_t idesc_qk = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(ATT_TK >> 3) << 17) | ((uint32_t)(ATT_PAIRS >> 4) << 24);
    const uint32_t idesc_pv = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(HD >> 3) << 17) | ((uint32_t)(ATT_PAIRS >> 4) << 24);
    const uint32_t el = elect_one();
    uint32_t n = 0;
    bool ok = true;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      ok = tc::mbar_wait(tc::smem_u32(bar), parity, p.status, p.spin_fast, p.spin_slow);
      ok = __all_sync(0xffffffffu, ok);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      return ok;
    };
    auto scores = [&](int t) {
      const uint32_t s = n % ATT_RING;
      if (!wait(&sh->kv_full[s], (n / ATT_RING) & 1u)) return;
      const uint32_t k_base = base + 2 * Q_BYTES + s * KV_BYTES, d = tmem + S_COL + (t & 1) * ATT_TK;
#pragma unroll
      for (int part = 0; part < 2; ++part)
#pragma unroll
        for (int s8 = 0; s8 < HD / 16; ++s8) {
          const uint64_t da = tc::make_smem_desc(base + part * Q_BYTES + (s8 >> 2) * (ATT_PAIRS * 128)) + (uint64_t)((s8 & 3) * 2);
          const uint64_t db = tc::make_smem_desc(k_base + (s8 >> 2) * (KV_BYTES / 2)) + (uint64_t)((s8 & 3) * 2);
          mma_ss(d, da, db, idesc_qk, part > 0 || s8 > 0, el);
        }
      commit_one(tc::smem_u32(&sh->kv_empty[s]), el);
      commit_one(tc::smem_u32(&sh->s_full[t & 1]), el);
      ++n;
    };
    if (nt > 0) scores(0);
    for (int t = 0; t < nt && ok; ++t) {
      if (t + 1 < nt) scores(t + 1);   // (buffer of tile t - 1: its P V was issued before, the tensor pipe keeps the order)
      if (!ok || !wait(&sh->p_full[t & 1], (t >> 1) & 1u)) break;
      const uint32_t s = n % ATT_RING;
      if (!wait(&sh->kv_full[s], (n / ATT_RING) & 1u)) break;
      const uint32_t v_base = base + 2 * Q_BYTES + s * KV_BYTES, a = tmem + S_COL + (t & 1) * ATT_TK;
      // V tile as the cache has it: key rows of 128 dims, the MN-major form of B (64-dim halves KV_BYTES / 2 apart)
      const uint64_t db = (tc::make_smem_desc(v_base) & ~(0x3FFFull << 16)) | ((uint64_t)(KV_BYTES / 2 / 16) << 16);
#pragma unroll
      for (int part = 0; part < 2; ++part)
#pragma unroll
        for (int s4 = 0; s4 < ATT_TK / 16; ++s4)
          mma_ts(tmem + O_COL, a + part * (ATT_TK / 2) + s4 * 8, db + (uint64_t)(s4 * 128), idesc_pv, t > 0 || part > 0 || s4 > 0, el);
      commit_one(tc::smem_u32(&sh->kv_empty[s]), el);
      commit_one(tc::smem_u32(&sh->o_done[t & 1]), el);
      ++n;
    }
    if (!ok) sh->abort = 1;
  } else {
    const int pp = pair0 + (int)threadIdx.x;
    const bool pv = pp < Pn;
    const int r = pv ? pp / Gq : 0, hq = kvh * Gq + (pv ? pp % Gq : 0);
    const int own_first = r / p.T * p.T;
    const uint32_t t_row = tmem + ((uint32_t)(warp * 32) << 16);
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int t = 0; t < nt; ++t) {
      ok = tc::mbar_wait(tc::smem_u32(&sh->s_full[t & 1]), (t >> 1) & 1u, p.status, p.spin_fast, p.spin_slow);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float s[ATT_TK];
      const uint32_t t_s = t_row + S_COL + (t & 1) * ATT_TK;
      {
        float a[32], c[32];
        tmem_ld<32>(t_s, a);
        tmem_ld<32>(t_s + 32, c);
        tmem_wait_ld();
#pragma unroll
        for (int k = 0; k < 32; ++k) { s[k] = a[k]; s[32 + k] = c[k]; }
      }
      // visible keys of the tile: [lo, hi)
      const int tt = t_lo + t;
      int lo = 0, hi = ATT_TK;
      if (tt < nt_c) {
        hi = min(ATT_TK, p.C - tt * ATT_TK);
      } else {
        const int y = own_lo + (tt - nt_c) * ATT_TK;
        lo = max(0, own_first - y);
        hi = min(ATT_TK, r + 1 - y);
      }
      if (!pv) hi = 0;
      if (__any_sync(0xffffffffu, lo > 0 || hi < ATT_TK)) {
#pragma unroll
        for (int k = 0; k < ATT_TK; ++k)
          if (k < lo || k >= hi) s[k] = -INFINITY;
      }
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int k = 0; k < ATT_TK; ++k) m4[k & 3] = fmaxf(m4[k & 3], s[k]);
      const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
      const bool grow = t > 0 && mx > m + 8.f;   // (also the first visible key of the row: m = -inf)
      if (t == 0) {
        m = mx;
      } else if (__any_sync(0xffffffffu, grow)) {
        // the outputs so far are rescaled: every P V issued so far (tile t - 1 is the last) has to be done
        ok = tc::mbar_wait(tc::smem_u32(&sh->o_done[(t - 1) & 1]), ((t - 1) >> 1) & 1u, p.status, p.spin_fast, p.spin_slow);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const float corr = grow ? exp2f(m - mx) : 1.f;
        if (grow) { l *= corr; m = mx; }
#pragma unroll 1
        for (int c = 0; c < HD; c += 32) {
          float o[32];
          tmem_ld<32>(t_row + O_COL + c, o);
          tmem_wait_ld();
          uint32_t u[32];
#pragma unroll
          for (int k = 0; k < 32; ++k) u[k] = __float_as_uint(o[k] * corr);
          tmem_st32(t_row + O_COL + c, u);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      }
      const float mm = m == -INFINITY ? 0.f : m;   // no visible key so far: all weights are exp2(-inf) = 0
      float r4[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t ph[ATT_TK / 2], pl[ATT_TK / 2];
#pragma unroll
      for (int k = 0; k < ATT_TK; k += 2) {
        const float a = ex2(s[k] - mm), c = ex2(s[k + 1] - mm);
        r4[(k >> 1) & 3] += a + c;
        split2(a, c, ph[k >> 1], pl[k >> 1]);
      }
      l += (r4[0] + r4[1]) + (r4[2] + r4[3]);
      tmem_st32(t_s, ph);
      tmem_st32(t_s + ATT_TK / 2, pl);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&sh->p_full[t & 1])) : "memory");
    }
    if (ok && nt > 0) {
      ok = tc::mbar_wait(tc::smem_u32(&sh->o_done[(nt - 1) & 1]), ((nt - 1) >> 1) & 1u, p.status, p.spin_fast, p.spin_slow);
      ok = __all_sync(0xffffffffu, ok);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    if (!ok) sh->abort = 1;
    if (ok) {
      const float inv = 1.0f / l;
      const long long idx = ((long long)r * p.nq + hq) * p.splits + split;
#pragma unroll 1
      for (int c = 0; c < HD; c += 32) {
        float o[32];
        if (nt > 0) {
          tmem_ld<32>(t_row + O_COL + c, o);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int k = 0; k < 32; ++k) o[k] = 0.f;
        }
        if (p.splits == 1) {
          bf16* dst = p.out + ((long long)r * p.nq + hq) * HD + c;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            st16b(dst + 8 * k, pack2(o[8 * k] * inv, o[8 * k + 1] * inv), pack2(o[8 * k + 2] * inv, o[8 * k + 3] * inv),
                  pack2(o[8 * k + 4] * inv, o[8 * k + 5] * inv), pack2(o[8 * k + 6] * inv, o[8 * k + 7] * inv), pv);
        } else {
#pragma unroll
          for (int k = 0; k < 4; ++k) st8(p.part_acc + idx * HD + c + 8 * k, o + 8 * k, true, pv);
        }
      }
      if (pv && p.splits > 1) p.part_ml[idx] = make_float2(m, l);
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (sh->abort)
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  if (warp == 5) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256u) : "memory");
  }
}

}  // namespace wide
}  // namespace clasp
