// kvr_split.cu -- full-context decode attention split over the rows (the
// KV-Rescue helper keeps its full cache, Sec. 3.1 / App. D): append the new
// row and compute Attn(q_t, C) (Eq. 1) over every cached row, with no
// importance scores and no eviction; and the same with scores for units that
// a prompt left long (the step before their first eviction).  bf16, head_dim
// 128, G <= 8.
//
// split_partial_kernel: grid (splits, units).  Each CTA takes a contiguous
//   chunk of a unit's rows and streams it through shared memory in 64-row
//   stages (two 128B-swizzled TMA boxes for K and two for V per stage,
//   double-buffered on mbarriers).  Each of the 4 warps owns one 16-row tile
//   per stage: QK^T and PV on bf16 mma.sync (P split hi + lo), with an online
//   softmax (running max and sum per query head).  The warps' states are
//   merged in shared memory and the CTA writes its (max, sum, unnormalised
//   output) to the workspace.
// long_step_kernel: grid (8, units), a cluster a unit: the same stream with
//   importance scores, for kvr_decode_attend_score over long units.
// split_combine_kernel: grid (units).  Merges the splits of a unit into the
//   output, then appends the new row to the cache (the partial kernels only
//   read the slab, so nothing races).
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include "kvr_internal.h"
#include "kvr_ptx.cuh"

namespace kvr {
namespace {

using namespace ptx;

constexpr int kRows = 64;                     // rows per stage
constexpr int kWarps = 4;                     // one 16-row tile each
constexpr int kStages = 2;
constexpr int kBox = kRows * 128;             // bytes of one 64-column box
constexpr int kStageBytes = 4 * kBox;         // K0, K1, V0, V1
constexpr int kQPitch = 272;
constexpr int kWsStride = 130;                // floats per (split, head)

struct SmemLayout {
  static constexpr int q = kStages * kStageBytes;
  static constexpr int ml = q + 8 * kQPitch;  // [warp][8] max, [warp][8] sum
  static constexpr int bytes = ml + 2 * kWarps * 8 * 4;
};

// Attention of the G query heads over rows [r0, r1) of one unit (len rows in
// the slab, the new row after them), r0 < r1.  The CTA's four warps leave
// their merged state with warp 0, which hands each value to put_o(g, d, sum)
// and put_ml(g, max, sum); kLogits: the scaled logits (base 2) also go to
// lg[row * G + g].  PV takes P as kTerms bf16 terms (2: 16 bits of mantissa, 3:
// all of fp32's).  False if a copy timed out (the error word is set and the
// copies in flight have landed).  (The kernel's parameters come as they are: as
// eight arguments the compiler put fewer loads in flight, 80 registers against
// 96, and the helper's step took 1,067 us instead of 1,059.)
template <bool kLogits, int kTerms, typename PutO, typename PutMl>
__device__ __forceinline__ bool attend_rows(const CUtensorMap &tmK, const CUtensorMap &tmV,
                                            const SplitParams &p, unsigned char *smem,
                                            uint64_t *full_bar, volatile int &s_abort,
                                            size_t ug, size_t krow, int len, int r0, int r1,
                                            float *lg, PutO put_o, PutMl put_ml) {
  const CacheView &c = p.c;
  const int G = c.G;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_st = (r1 - r0 + kRows - 1) / kRows;
  const int row0 = (int)(ug * (size_t)c.cap) + r0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) mbar_init(smem_u32(&full_bar[s]), 1);
    s_abort = 0;
    fence_mbar_init();
  }
  // Query rows (zero beyond G) with plain loads; bounded by 8 x 256 bytes.
  {
    const int4 *qg = reinterpret_cast<const int4 *>(p.q + krow * G * 128);
    for (int i = threadIdx.x; i < 8 * 16; i += blockDim.x) {
      const int g = i >> 4, ch = i & 15;
      *reinterpret_cast<int4 *>(smem + SmemLayout::q + g * kQPitch + ch * 16) =
          g < G ? qg[g * 16 + ch] : make_int4(0, 0, 0, 0);
    }
  }
  __syncthreads();
  auto issue = [&](int st) {
    const uint32_t b = smem_u32(&full_bar[st % kStages]);
    const uint32_t dst = smem_u32(smem + (st % kStages) * kStageBytes);
    mbar_expect_tx(b, kStageBytes);
    const int y = row0 + st * kRows;
    tma_load_2d(dst, &tmK, 0, y, b);
    tma_load_2d(dst + kBox, &tmK, 64, y, b);
    tma_load_2d(dst + 2 * kBox, &tmV, 0, y, b);
    tma_load_2d(dst + 3 * kBox, &tmV, 64, y, b);
  };
  if (threadIdx.x == 0)
    for (int st = 0; st < min(kStages, n_st); ++st) issue(st);

  uint32_t qb[8][2];
  {
    const uint32_t qa = smem_u32(smem + SmemLayout::q) + (lane & 7) * kQPitch +
                        (lane >> 3) * 16;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      ldsm_x4(qa + i * 64, qb[2 * i][0], qb[2 * i][1], qb[2 * i + 1][0],
              qb[2 * i + 1][1]);
  }
  const int r0l = lane >> 2, c2 = (lane & 3) * 2;
  float m0 = -INFINITY, m1 = -INFINITY;  // running max of columns c2, c2+1
  float l0 = 0.f, l1 = 0.f;              // this lane's share of the sums
  float o[8][4];
#pragma unroll
  for (int mt = 0; mt < 8; ++mt) o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f;

  for (int st = 0; st < n_st; ++st) {
    const int buf = st % kStages;
    if (!mbar_wait(smem_u32(&full_bar[buf]), (uint32_t)(st / kStages) & 1u,
                   &s_abort)) {
      if (lane == 0) {
        atomicOr(c.err, ERR_TIMEOUT);
        s_abort = 1;
      }
      break;
    }
    unsigned char *K0 = smem + buf * kStageBytes, *K1 = K0 + kBox;
    unsigned char *V0 = K0 + 2 * kBox, *V1 = K0 + 3 * kBox;
    const int base = r0 + st * kRows;  // unit row of stage row 0
    const int t0 = warp * 16;          // this warp's tile in the stage
    // The new row (unit row len) comes from the inputs; rows at or beyond
    // the chunk end are masked and their V zeroed (they may hold anything).
    {
      const int rn = len - base;
      if (rn >= t0 && rn < t0 + 16) {
        const int chunk16 = lane & 15, half = chunk16 >> 3, cc = chunk16 & 7;
        const uint32_t off = rn * 128 + ((cc ^ (rn & 7)) << 4);
        unsigned char *dst = lane < 16 ? (half ? K1 : K0) : (half ? V1 : V0);
        const __nv_bfloat16 *src = (lane < 16 ? p.k_new : p.v_new) + krow * 128;
        *reinterpret_cast<int4 *>(dst + off) =
            reinterpret_cast<const int4 *>(src)[chunk16];
      }
      const int lo = max(t0, r1 - base);
      for (int i = lane; i < (t0 + 16 - lo) * 16; i += 32) {
        const int r = lo + (i >> 4), c16 = i & 15;
        if (r >= t0)
          *reinterpret_cast<int4 *>((c16 < 8 ? V0 : V1) + r * 128 +
                                    (c16 & 7) * 16) = make_int4(0, 0, 0, 0);
      }
    }
    __syncwarp();
    if (base + t0 < r1) {
      float s[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
      {
        const int row = t0 + (lane & 7) + ((lane >> 3) & 1) * 8;
        const uint32_t b0 = smem_u32(K0) + row * 128, b1 = smem_u32(K1) + row * 128;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
          const int cc = ((ks & 3) << 1) + (lane >> 4);
          const uint32_t addr = (ks >> 2 ? b1 : b0) + ((cc ^ (row & 7)) << 4);
          uint32_t a0, a1, a2, a3;
          ldsm_x4(addr, a0, a1, a2, a3);
          if (ks & 1) mma_bf16(s2, a0, a1, a2, a3, qb[ks][0], qb[ks][1]);
          else mma_bf16(s, a0, a1, a2, a3, qb[ks][0], qb[ks][1]);
        }
      }
      const int ra = base + t0 + r0l, rb = ra + 8;
      s[0] = ra < r1 ? (s[0] + s2[0]) * p.scale_log2e : -INFINITY;
      s[1] = ra < r1 ? (s[1] + s2[1]) * p.scale_log2e : -INFINITY;
      s[2] = rb < r1 ? (s[2] + s2[2]) * p.scale_log2e : -INFINITY;
      s[3] = rb < r1 ? (s[3] + s2[3]) * p.scale_log2e : -INFINITY;
      if constexpr (kLogits) {
        if (c2 < G) {
          if (ra < r1) lg[(size_t)ra * G + c2] = s[0];
          if (rb < r1) lg[(size_t)rb * G + c2] = s[2];
        }
        if (c2 + 1 < G) {
          if (ra < r1) lg[(size_t)ra * G + c2 + 1] = s[1];
          if (rb < r1) lg[(size_t)rb * G + c2 + 1] = s[3];
        }
      }
      float x0 = fmaxf(s[0], s[2]), x1 = fmaxf(s[1], s[3]);
#pragma unroll
      for (int off = 4; off < 32; off <<= 1) {
        x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, off));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, off));
      }
      const float n0 = fmaxf(m0, x0), n1 = fmaxf(m1, x1);  // finite: row ra valid
      const float a0 = exp2f(m0 - n0), a1 = exp2f(m1 - n1);
      m0 = n0;
      m1 = n1;
      s[0] = exp2f(s[0] - m0);
      s[1] = exp2f(s[1] - m1);
      s[2] = exp2f(s[2] - m0);
      s[3] = exp2f(s[3] - m1);
      l0 = l0 * a0 + s[0] + s[2];
      l1 = l1 * a1 + s[1] + s[3];
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        o[mt][0] *= a0;
        o[mt][2] *= a0;
        o[mt][1] *= a1;
        o[mt][3] *= a1;
      }
      const uint32_t h0 = pack_bf16(s[0], s[1]), h1 = pack_bf16(s[2], s[3]);
      const __nv_bfloat162 hb0 = *reinterpret_cast<const __nv_bfloat162 *>(&h0);
      const __nv_bfloat162 hb1 = *reinterpret_cast<const __nv_bfloat162 *>(&h1);
      const uint32_t bp0 = movm_t(h0), bp1 = movm_t(h1);
      // (the remainders are exact)
      const float e0 = s[0] - __low2float(hb0), e1 = s[1] - __high2float(hb0);
      const float e2 = s[2] - __low2float(hb1), e3 = s[3] - __high2float(hb1);
      const uint32_t g0 = pack_bf16(e0, e1), g1 = pack_bf16(e2, e3);
      const uint32_t bl0 = movm_t(g0), bl1 = movm_t(g1);
      uint32_t bm0 = 0u, bm1 = 0u;
      if constexpr (kTerms == 3) {
        const __nv_bfloat162 lb0 = *reinterpret_cast<const __nv_bfloat162 *>(&g0);
        const __nv_bfloat162 lb1 = *reinterpret_cast<const __nv_bfloat162 *>(&g1);
        bm0 = movm_t(pack_bf16(e0 - __low2float(lb0), e1 - __high2float(lb0)));
        bm1 = movm_t(pack_bf16(e2 - __low2float(lb1), e3 - __high2float(lb1)));
      }
      const int row = t0 + (lane & 7) + ((lane >> 4) << 3);
      const uint32_t b0 = smem_u32(V0) + row * 128, b1 = smem_u32(V1) + row * 128;
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        const int c16 = 2 * mt + ((lane >> 3) & 1);
        const uint32_t addr = (c16 >> 3 ? b1 : b0) + (((c16 & 7) ^ (row & 7)) << 4);
        uint32_t v0, v1, v2, v3;
        ldsm_x4_t(addr, v0, v1, v2, v3);
        mma_bf16(o[mt], v0, v1, v2, v3, bp0, bp1);
        mma_bf16(o[mt], v0, v1, v2, v3, bl0, bl1);
        if constexpr (kTerms == 3) mma_bf16(o[mt], v0, v1, v2, v3, bm0, bm1);
      }
    }
    // Refill this buffer once every warp is done with it.
    fence_proxy_async();
    __syncthreads();
    if (threadIdx.x == 0 && st + kStages < n_st) issue(st + kStages);
  }
  __syncthreads();
  if (s_abort) {  // drain copies still landing in our buffers (bounded)
    if (threadIdx.x == 0) {
      volatile int never = 0;
      for (int st = 0; st < n_st; ++st)
        mbar_wait(smem_u32(&full_bar[st % kStages]), (uint32_t)(st / kStages) & 1u,
                  &never);
    }
    __syncthreads();
    return false;
  }

  // Merge the four warps: common max per head, rescaled sums and outputs.
#pragma unroll
  for (int off = 4; off < 32; off <<= 1) {
    l0 += __shfl_xor_sync(0xffffffffu, l0, off);
    l1 += __shfl_xor_sync(0xffffffffu, l1, off);
  }
  float *ML = reinterpret_cast<float *>(smem + SmemLayout::ml);
  if (lane < 4) {
    ML[warp * 8 + c2] = m0;
    ML[warp * 8 + c2 + 1] = m1;
  }
  __syncthreads();
  float M0 = -INFINITY, M1 = -INFINITY;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    M0 = fmaxf(M0, ML[w * 8 + c2]);
    M1 = fmaxf(M1, ML[w * 8 + c2 + 1]);
  }
  const float f0 = m0 == -INFINITY ? 0.f : exp2f(m0 - M0);
  const float f1 = m1 == -INFINITY ? 0.f : exp2f(m1 - M1);
  float *XO = reinterpret_cast<float *>(smem);  // [warp][mt][4][32]
#pragma unroll
  for (int mt = 0; mt < 8; ++mt) {
    XO[((warp * 8 + mt) * 4 + 0) * 32 + lane] = o[mt][0] * f0;
    XO[((warp * 8 + mt) * 4 + 1) * 32 + lane] = o[mt][1] * f1;
    XO[((warp * 8 + mt) * 4 + 2) * 32 + lane] = o[mt][2] * f0;
    XO[((warp * 8 + mt) * 4 + 3) * 32 + lane] = o[mt][3] * f1;
  }
  if (lane < 4) {
    ML[32 + warp * 8 + c2] = l0 * f0;
    ML[32 + warp * 8 + c2 + 1] = l1 * f1;
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) sum += XO[((w * 8 + mt) * 4 + e) * 32 + lane];
        const int g = c2 + (e & 1), d = 16 * mt + r0l + 8 * (e >> 1);
        if (g < G) put_o(g, d, sum);
      }
    }
    if (lane < 4) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int g = c2 + e;
        if (g < G) {
          float L = 0.f;
#pragma unroll
          for (int w = 0; w < kWarps; ++w) L += ML[32 + w * 8 + g];
          put_ml(g, e ? M1 : M0, L);
        }
      }
    }
  }
  return true;
}

__global__ void __launch_bounds__(32 * kWarps)
    split_partial_kernel(const __grid_constant__ CUtensorMap tmK,
                         const __grid_constant__ CUtensorMap tmV,
                         const SplitParams p) {
  pdl_begin();
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kStages];
  __shared__ volatile int s_abort;
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const CacheView &c = p.c;
  const int G = c.G;
  const int split = blockIdx.x, idx = blockIdx.y;
  const int h = idx % c.H, lr = (idx / c.H) % p.nl, sq = idx / (c.H * p.nl);
  const size_t ug = ((size_t)sq * c.L + p.lb + lr) * c.H + h;
  const size_t krow = ((size_t)sq * p.nl + lr) * c.H + h;
  const int len = c.state[4 * ug];
  const int n = len + 1;
  int chunk = (n + p.n_splits - 1) / p.n_splits;
  chunk = (chunk + kRows - 1) / kRows * kRows;
  const int r0 = split * chunk, r1 = min(n, r0 + chunk);
  float *ws = p.ws + (((size_t)idx * p.n_splits + split) * G) * kWsStride;
  if (r0 >= r1) {  // an empty split contributes nothing
    for (int g = threadIdx.x; g < G; g += blockDim.x) {
      ws[g * kWsStride] = -INFINITY;
      ws[g * kWsStride + 1] = 0.f;
    }
    return;
  }
  attend_rows<false, 2>(
      tmK, tmV, p, smem, full_bar, s_abort, ug, krow, len, r0, r1, nullptr,
      [&](int g, int d, float x) { ws[g * kWsStride + 2 + d] = x; },
      [&](int g, float M, float L) {
        ws[g * kWsStride] = M;
        ws[g * kWsStride + 1] = L;
      });
}

template <typename O>
__global__ void __launch_bounds__(128) split_combine_kernel(const SplitParams p,
                                                            void *out) {
  pdl_begin();
  const CacheView &c = p.c;
  const int G = c.G, idx = blockIdx.x;
  const int h = idx % c.H, lr = (idx / c.H) % p.nl, sq = idx / (c.H * p.nl);
  const size_t ug = ((size_t)sq * c.L + p.lb + lr) * c.H + h;
  const size_t krow = ((size_t)sq * p.nl + lr) * c.H + h;
  const float *ws = p.ws + (size_t)idx * p.n_splits * G * kWsStride;
  const int d = threadIdx.x;  // 128 threads, one head-dim column each
  O *og = reinterpret_cast<O *>(out) + krow * G * 128;
  for (int g = 0; g < G; ++g) {
    float M = -INFINITY;
    for (int s = 0; s < p.n_splits; ++s) M = fmaxf(M, ws[(s * G + g) * kWsStride]);
    float L = 0.f, acc = 0.f;
    for (int s = 0; s < p.n_splits; ++s) {
      const float *w = ws + (s * G + g) * kWsStride;
      if (w[0] == -INFINITY) continue;  // empty split: its outputs are unset
      const float f = exp2f(w[0] - M);
      L += w[1] * f;
      acc += w[2 + d] * f;
    }
    if (d == 0 && !(L >= 1.f && L < INFINITY)) atomicOr(c.err, ERR_NONFINITE);
    const float v = acc / L;
    if constexpr (sizeof(O) == 2) og[g * 128 + d] = __float2bfloat16_rn(v);
    else og[g * 128 + d] = v;
  }
  // Append the new row now that every split has read the slab.
  const int len = c.state[4 * ug], t = c.state[4 * ug + 1];
  __nv_bfloat16 *K = reinterpret_cast<__nv_bfloat16 *>(c.K) + (ug * c.cap + len) * 128;
  __nv_bfloat16 *V = reinterpret_cast<__nv_bfloat16 *>(c.V) + (ug * c.cap + len) * 128;
  K[d] = p.k_new[krow * 128 + d];
  V[d] = p.v_new[krow * 128 + d];
  __syncthreads();  // every thread has read the state before it changes
  if (d == 0) {
    c.pos[ug * c.sstride + len] = t;
    c.score[ug * c.sstride + len] = 0.f;
    c.state[4 * ug] = len + 1;
    c.state[4 * ug + 1] = t + 1;
    c.state[4 * ug + 2] = 0;  // the R-KV key sum no longer matches
  }
}

// ---- the scoring step over long units ------------------------------------------

constexpr int kCluster = 8;         // CTAs a cluster, at most
constexpr int kClusterRows = 1024;  // rows a CTA should have

__device__ __forceinline__ void cluster_sync() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
          : "memory");
}
// A float of the same shared-memory variable in CTA `rank` of the cluster.
__device__ __forceinline__ float peer_float(const float *v, int rank) {
  uint32_t a;
  float x;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(v)), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(a) : "memory");
  return x;
}

// Steps 1-3 of a decode step (append, attend, accumulate scores) for units
// too long for one CTA: one cluster of up to eight CTAs a unit, a contiguous
// share of the rows each, K and V read once.  The CTAs' softmax states and partial
// outputs meet in distributed shared memory, so nothing but the logits (28
// bytes a row of 512, in the cache's scratch, from which each CTA then forms
// its rows' exact probabilities) goes through global memory.  It is bound by
// the K and V stream.  One CTA a unit instead (attend_score_kernel) leaves
// the step waiting for the longest unit: 7B, four prompts of 700 to 16,384
// rows, took 6.03 ms, this 0.31 (4.5 TB/s; four of 16,384 rows, 5.4).  What is
// left is the score pass after the merge (0.04 ms: each CTA waits for its
// logits from L2) and the ends of the clusters.
template <typename O>
__global__ void __launch_bounds__(32 * kWarps)
    long_step_kernel(const __grid_constant__ CUtensorMap tmK,
                     const __grid_constant__ CUtensorMap tmV, const SplitParams p,
                     const __grid_constant__ SeqOrder order, O *out) {
  pdl_begin();
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[kStages];
  __shared__ volatile int s_abort;
  __shared__ float s_o[8 * 128], s_m[8], s_l[8];  // this CTA's partial state
  __shared__ float s_f[kCluster][8], s_M[8], s_iL[8];
  const int nc = gridDim.x;  // CTAs of the unit's cluster: 1, 2, 4 or 8
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const CacheView &c = p.c;
  const int G = c.G, tid = threadIdx.x;
  const int rank = blockIdx.x, idx = blockIdx.y;
  const int h = idx % c.H, lr = (idx / c.H) % p.nl;
  int sq = idx / (c.H * p.nl);
  if (c.S <= kMaxOrder) sq = order.seq[sq];
  const size_t ug = ((size_t)sq * c.L + p.lb + lr) * c.H + h;
  const size_t krow = ((size_t)sq * p.nl + lr) * c.H + h;
  const int len = c.state[4 * ug], newest = c.state[4 * ug + 1];
  const int n = len + 1;
  const bool fits = len >= 0 && n <= c.cap;
  if (!fits && tid == 0 && rank == 0) atomicOr(c.err, ERR_CAPACITY);
  int chunk = (n + nc - 1) / nc;
  chunk = (chunk + kRows - 1) / kRows * kRows;
  const int r0 = rank * chunk, r1 = fits ? min(n, r0 + chunk) : 0;
  float *lg = c.logits + ug * (size_t)G * c.cap;
  for (int i = tid; i < 8 * 128; i += 32 * kWarps) s_o[i] = 0.f;
  if (tid < 8) {
    s_m[tid] = -INFINITY;
    s_l[tid] = 0.f;
  }
  __syncthreads();
  if (r0 < r1)
    // (P whole, as the generic kernel has it: 789 us against 786 for the load
    // and step of the prompts above with two terms, which bf16 outputs hide.)
    attend_rows<true, 3>(
        tmK, tmV, p, smem, full_bar, s_abort, ug, krow, len, r0, r1, lg,
        [&](int g, int d, float x) { s_o[g * 128 + d] = x; },
        [&](int g, float M, float L) {
          s_m[g] = M;
          s_l[g] = L;
        });
  // (A CTA whose copies timed out takes part with what it has: the error
  // word says that the unit is undefined.)
  __syncthreads();
  cluster_sync();
  if (tid < 8 * nc) {
    const int g = tid & 7, k = tid >> 3;
    s_f[k][g] = peer_float(&s_m[g], k);
  }
  __syncthreads();
  if (tid < 8) {
    float M = -INFINITY, L = 0.f;
    for (int k = 0; k < nc; ++k) M = fmaxf(M, s_f[k][tid]);
    for (int k = 0; k < nc; ++k) {
      const float f = s_f[k][tid] == -INFINITY ? 0.f : exp2f(s_f[k][tid] - M);
      L += peer_float(&s_l[tid], k) * f;
      s_f[k][tid] = f;
    }
    s_M[tid] = M;
    s_iL[tid] = 1.f / L;
    if (rank == 0 && fits && tid < G && !(L >= 1.f && L < INFINITY))
      atomicOr(c.err, ERR_NONFINITE);
  }
  __syncthreads();
  // The CTAs take the heads' outputs in turn.
  for (int g = rank; fits && g < G; g += nc) {
    float acc = 0.f;
    for (int k = 0; k < nc; ++k) acc += peer_float(&s_o[g * 128 + tid], k) * s_f[k][g];
    const float v = acc * s_iL[g];
    O *og = out + (krow * G + g) * 128;
    if constexpr (sizeof(O) == 2) og[tid] = __float2bfloat16_rn(v);
    else og[tid] = v;
  }
  // The rows' probabilities, and the head mean onto their scores.
  const float inv_g = 1.f / (float)G;
  float *su = c.score + ug * (size_t)c.sstride;
  constexpr int kAhead = 4;  // rows a thread has in flight
  for (int i0 = r0 + tid; i0 < r1; i0 += kAhead * 32 * kWarps) {
    float x[kAhead][8], sc[kAhead];
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      const int i = i0 + k * 32 * kWarps;
      sc[k] = i < len && i < r1 ? su[i] : 0.f;  // the appended row starts at zero
#pragma unroll
      for (int g = 0; g < 8; ++g) x[k][g] = g < G && i < r1 ? lg[(size_t)i * G + g] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      const int i = i0 + k * 32 * kWarps;
      float acc = 0.f;
#pragma unroll
      for (int g = 0; g < 8; ++g)
        if (g < G) acc += exp2f(x[k][g] - s_M[g]) * s_iL[g];
      if (i < r1) su[i] = sc[k] + acc * inv_g;
    }
  }
  // The CTA with the new row writes it to its slot (every read of that slot
  // was masked or replaced).
  if (r0 <= len && len < r1) {
    const size_t dst = (ug * c.cap + len) * 128;
    reinterpret_cast<__nv_bfloat16 *>(c.K)[dst + tid] = p.k_new[krow * 128 + tid];
    reinterpret_cast<__nv_bfloat16 *>(c.V)[dst + tid] = p.v_new[krow * 128 + tid];
    if (tid == 0) c.pos[ug * (size_t)c.sstride + len] = newest;
  }
  // Every CTA has read its peers' shared memory and the unit's state.
  __syncthreads();
  cluster_sync();
  if (rank == 0 && tid == 0 && fits) {
    c.state[4 * ug] = n;
    c.state[4 * ug + 1] = newest + 1;
    c.state[4 * ug + 2] = 0;  // the R-KV key sum no longer matches
  }
}

}  // namespace

size_t split_workspace_bytes(const CacheView &c, int nl, int n_splits) {
  return (size_t)c.S * nl * c.H * n_splits * c.G * kWsStride * sizeof(float);
}

int split_rows_per_stage() { return kRows; }

cudaError_t launch_split_attend(const CUtensorMap &tmK, const CUtensorMap &tmV,
                                const SplitParams &p, void *out,
                                cudaStream_t st) {
  const int smem = SmemLayout::bytes + 1024;
  cudaError_t e = cudaFuncSetAttribute(
      split_partial_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int units = p.c.S * p.nl * p.c.H;
  e = launch_pdl(split_partial_kernel, dim3(p.n_splits, units),
                 dim3(32 * kWarps), smem, st, tmK, tmV, p);
  if (e != cudaSuccess) return e;
  if (p.c.out_bf16)
    return launch_pdl(split_combine_kernel<__nv_bfloat16>, dim3(units),
                      dim3(128), 0, st, p, out);
  return launch_pdl(split_combine_kernel<float>, dim3(units), dim3(128), 0, st,
                    p, out);
}

cudaError_t launch_long_step(const CUtensorMap &tmK, const CUtensorMap &tmV,
                             const SplitParams &p, const SeqOrder &order, int max_rows,
                             int sms, void *out, cudaStream_t st) {
  const int smem = SmemLayout::bytes + 1024;
  cudaLaunchConfig_t cfg = {};
  // Eight CTAs a unit only where its rows or the launch's width ask for them:
  // each has a start and an end outside the stream (two prompts of 2,500 and
  // 3,000 rows, 7B: 102 us with eight, 76 with four; one of 16,384: 221 and
  // 224).
  const int units = p.c.S * p.nl * p.c.H;
  int nc = 1;
  const int fill = 8 * sms / 3;  // about one for each of an SM's three places
  while (nc < kCluster && (max_rows > nc * kClusterRows * 2 || units * nc < fill)) nc *= 2;
  cfg.gridDim = dim3(nc, units);
  cfg.blockDim = dim3(32 * kWarps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = nc;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  auto run = [&](auto kern, auto *o) {
    const cudaError_t e = cudaFuncSetAttribute(
        kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, kern, tmK, tmV, p, order, o);
  };
  return p.c.out_bf16
             ? run(long_step_kernel<__nv_bfloat16>, static_cast<__nv_bfloat16 *>(out))
             : run(long_step_kernel<float>, static_cast<float *>(out));
}

}  // namespace kvr
