// kvr_fork_tile.cu -- the candidate step of stepwise best-of-N (Sec. 2.2 Eq. 2,
// App. C) as tiles on 5th-generation tensor cores: N candidates share the
// parent's live rows as a read-only prefix and each has a private tail.  Per
// candidate: append + Attn(q_t, C) (Eq. 1) over prefix + tail + new row, and
// the accumulated attention (Sec. 2.1, mean over the G heads) of every row.
// bf16, head_dim 128, N <= 8, G <= 8, every unit of the call at the same tail
// length.
//
// Design (GB300, sm_103a).  The N x G query rows of a unit are one 128-row
// tile (two candidates in the first 2 G lanes of each 32-lane quarter), and
// its keys come in blocks of up to 128: the prefix, which all candidates see,
// then T = 16 (8 / N) rows of every candidate's tail side by side, of which a
// row sees its own.  What the mask throws away costs little (a 128-key block
// is 0.3 us of tensor time), while each K and V row is read and each MMA
// operand formed once for all candidates; one warp a candidate on mma.sync
// (kvr_fork_batch.cu) pays both per candidate and is bound by its instruction
// latencies.  72B geometry, 4 sequences, N = 8, 72 + up to 16 rows: 108 us a
// token against 150; what bounds it is the chain of a unit's steps, about 2
// to 4 thousand cycles each for two units an SM.  Per unit: S = Q K^T, online
// softmax, O += P V block by block (P as two bf16 terms in tensor memory), then
// a second contraction with the keys on the lanes for the scores, as in
// kvr_absorb_long.cu: a row's sum over a candidate's heads is a sum inside one
// thread, and its probabilities are exact because the normalisers are known.
//  - Persistent, two CTAs an SM (256 TMEM columns, 101 KB each), a unit at a
//    time; one CTA's waits are the other's tensor time.  Eight softmax warps
//    (two for each 32 lanes, half of a block's columns each), a loading and an
//    issuing warp.
//  - The tail maps end at the call's tail length, so TMA zero-fills the rows
//    past it; the issuing warp puts the new rows, staged in shared memory,
//    into their block, and zeroes V rows past the prefix.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include "kvr_internal.h"
#include "kvr_tmem.cuh"

namespace kvr {
namespace {

using namespace ptx;

constexpr int kBlk = 128;          // keys a block; rows of the query tile
constexpr int kHalf = kBlk * 128;  // bytes of a 64-column half of a block
constexpr int kTile = 2 * kHalf;
constexpr int kBox = 32;           // slab rows a prefix box
constexpr int kMaxCand = 8;
constexpr int kThr = 320, kCols = 256;
constexpr int kNew = 2 * kMaxCand * 256;  // the new k rows, then the new v rows
constexpr int kSmem = 3 * kTile + 2 * kNew + 1024;
static_assert(kSmem + 4096 <= 113 * 1024, "two CTAs an SM, with the static variables");
constexpr float kLazy = 8.f;  // as in kvr_absorb_long.cu
constexpr uint32_t kGaveUp = 0x7FBADBADu;

__host__ __device__ inline int tail_rows(int N) { return 16 * (8 / N); }

struct TileUnit {
  size_t ug, row0;  // cache unit; unit row of the call ([S][nl][H])
  int np, nPB, nb;  // prefix rows, prefix blocks, blocks
};

__device__ __forceinline__ bool tile_unit(const ForkTileParams &p, int i, int nTB, TileUnit &u) {
  const CacheView &c = p.f.p;
  const int h = i % c.H, lr = (i / c.H) % p.nl, sq = i / (c.H * p.nl);
  u.ug = ((size_t)sq * c.L + p.lb + lr) * c.H + h;
  u.row0 = (size_t)i;
  u.np = c.state[4 * u.ug];
  u.nPB = (u.np + kBlk - 1) / kBlk;
  u.nb = u.nPB + nTB;
  return u.np >= 0 && u.np <= c.cap;
}

// Outputs c0 .. c0 + 63 of a candidate's query head from the rows it sees: the
// prefix, its own tail and its new row.
template <bool kOutBf16>
__device__ __noinline__ void outputs_alone(const ForkTileParams &p, int i, int cand, int g,
                                           int c0, float ref, float inv) {
  using B = __nv_bfloat16;
  const ForkView &f = p.f;
  const CacheView &c = f.p;
  const size_t units = (size_t)c.S * c.L * c.H, at = (size_t)cand * c.S * p.nl * c.H + i;
  TileUnit u;
  tile_unit(p, i, 0, u);
  unsigned char *orow = reinterpret_cast<unsigned char *>(p.out) +
                        ((at * c.G + g) * 128 + c0) * (kOutBf16 ? 2 : 4);
  const size_t pre = u.ug * (size_t)c.cap * 128;
  const size_t own = ((size_t)cand * units + u.ug) * (size_t)f.tcap * 128;
  const B *q = p.q + (at * c.G + g) * 128;
#pragma unroll 1
  for (int k = 0; k < 2; ++k) {
    float o[32];
    for (int x = 0; x < 32; ++x) o[x] = 0.f;
#pragma unroll 1
    for (int part = 0; part < 3; ++part) {
      const B *K = part == 0   ? reinterpret_cast<const B *>(c.K) + pre
                   : part == 1 ? reinterpret_cast<const B *>(f.TK) + own
                               : p.k_new + at * 128;
      const B *V = part == 0   ? reinterpret_cast<const B *>(c.V) + pre
                   : part == 1 ? reinterpret_cast<const B *>(f.TV) + own
                               : p.v_new + at * 128;
      attend_row(q, K, V, part == 0 ? u.np : part == 1 ? p.nt : 1, c0 + 32 * k, p.scale_log2e,
                 ref, o);
    }
    for (int x = 0; x < 16; ++x) {
      const float a = o[2 * x] * inv, b = o[2 * x + 1] * inv;
      if (kOutBf16) reinterpret_cast<uint32_t *>(orow + 64 * k)[x] = pack_bf16(a, b);
      else reinterpret_cast<float2 *>(orow + 128 * k)[x] = make_float2(a, b);
    }
  }
}

template <bool kOutBf16>
__global__ void __launch_bounds__(kThr, 2)
    fork_tile_kernel(const __grid_constant__ ForkTileParams p,
                     const __grid_constant__ CUtensorMap tmK,
                     const __grid_constant__ CUtensorMap tmV,
                     const __grid_constant__ CUtensorMap tmTK,
                     const __grid_constant__ CUtensorMap tmTV,
                     const __grid_constant__ CUtensorMap tmQ, int n_units) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  __shared__ float s_x[2][kBlk];              // what a row's two threads tell each other
  __shared__ __align__(16) float2 s_norm[kBlk];  // -reference and 1 / sum of each query row
  __shared__ __align__(8) uint64_t b_qfull[2], b_qfree[2], b_kfull, b_kfree, b_vfull, b_vfree, b_s,
      b_p, b_o, b_ref, b_sfree, b_drain;
  unsigned char *smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const uint32_t aQ = smem_u32(smem), aK = aQ + kTile, aV = aK + kTile;
  unsigned char *stage = smem + 3 * kTile;
  const ForkView &f = p.f;
  const CacheView &c = f.p;
  const int G = c.G, N = f.N, T = tail_rows(N), nt = p.nt, nTB = nt / T + 1;
  const int pairs = (N + 1) / 2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t units = (size_t)c.S * c.L * c.H, per = (size_t)n_units;
  volatile int *abort = &s_abort;
  // A whole warp's bounded wait for completion n of a barrier.
  auto wait_warp = [&](uint64_t &bar, int n) {
    return __all_sync(0xffffffffu, mbar_wait_idle(smem_u32(&bar), (uint32_t)(n & 1), abort)) != 0;
  };
  if (warp == 8) tmem_alloc(smem_u32(&s_tmem), kCols);
  if (tid == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&b_qfull[b]), 1);
      mbar_init(smem_u32(&b_qfree[b]), 1 + 8);  // the contractions; the softmax warps
    }
    mbar_init(smem_u32(&b_kfull), 1);
    mbar_init(smem_u32(&b_kfree), 1);
    mbar_init(smem_u32(&b_vfull), 1);
    mbar_init(smem_u32(&b_vfree), 1);
    mbar_init(smem_u32(&b_s), 1);
    mbar_init(smem_u32(&b_p), 8);
    mbar_init(smem_u32(&b_o), 1);
    mbar_init(smem_u32(&b_ref), 8);
    mbar_init(smem_u32(&b_sfree), 8);
    mbar_init(smem_u32(&b_drain), 1);
    s_abort = 0;
    fence_mbar_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  const uint32_t tm = s_tmem, tmO = tm + kBlk;

  if (warp == 8) {
    // Producer: one thread issues every load, in the order they are used: K
    // and V block by block, then, for the scores, K again, into the V buffer:
    // the next unit's first keys land in the other meanwhile.
    if (lane == 0) {
      prefetch_tmap(&tmK);
      prefetch_tmap(&tmV);
      prefetch_tmap(&tmTK);
      prefetch_tmap(&tmTV);
      prefetch_tmap(&tmQ);
      const uint32_t q_bytes = (uint32_t)(pairs * 2 * 2 * G * 128 + N * 512);
      int nq = 0, nk = 0, nv = 0;
      bool ok = true;
      // Rows of block j, keys or values, into the K or the V buffer.
      auto load_block = [&](bool kbuf, bool k, const TileUnit &u, int j) {
        int &n = kbuf ? nk : nv;
        if (n > 0)
          ok = mbar_wait_idle(smem_u32(kbuf ? &b_kfree : &b_vfree), (uint32_t)((n - 1) & 1), abort);
        if (!ok) return;
        ++n;
        const uint32_t bar = smem_u32(kbuf ? &b_kfull : &b_vfull), dst = kbuf ? aK : aV;
        if (j < u.nPB) {
          const int rows = min(kBlk, u.np - j * kBlk), nbox = (rows + kBox - 1) / kBox;
          const int row = (int)(u.ug * (size_t)c.cap) + j * kBlk;
          mbar_expect_tx(bar, (uint32_t)nbox * 2 * kBox * 128);
          for (int b = 0; b < nbox; ++b)
            for (int hf = 0; hf < 2; ++hf)
              tma_load_2d(dst + hf * kHalf + b * kBox * 128, k ? &tmK : &tmV, 64 * hf,
                          row + b * kBox, bar);
        } else {
          mbar_expect_tx(bar, (uint32_t)(N * T) * 256u);
          for (int hf = 0; hf < 2; ++hf)
            tma_load_4d(dst + hf * kHalf, k ? &tmTK : &tmTV, 64 * hf, (j - u.nPB) * T, (int)u.ug,
                        0, bar);
        }
      };
      // The queries and new rows of unit i, once: into the half of the tile
      // that the unit before last has left.
      int q_unit = -1;
      auto load_q = [&](int i) {
        if (q_unit >= i) return;
        const int b = nq & 1;
        if (nq > 1) ok = mbar_wait_idle(smem_u32(&b_qfree[b]), (uint32_t)((nq / 2 - 1) & 1), abort);
        if (!ok) return;
        const uint32_t bar = smem_u32(&b_qfull[b]), st = smem_u32(stage) + b * kNew;
        mbar_expect_tx(bar, q_bytes);
        for (int pr = 0; pr < pairs; ++pr)
          for (int hf = 0; hf < 2; ++hf)
            tma_load_4d(aQ + hf * kHalf + (pr * 32 + 16 * b) * 128, &tmQ, 64 * hf, 0, i, 2 * pr,
                        bar);
        for (int cd = 0; cd < N; ++cd) {
          const size_t src = ((size_t)cd * per + i) * 128;
          bulk_load(st + cd * 256, p.k_new + src, 256, bar);
          bulk_load(st + (kMaxCand + cd) * 256, p.v_new + src, 256, bar);
        }
        ++nq;
        q_unit = i;
      };
      // The next unit of this CTA (units with impossible lengths are skipped
      // by every role).
      auto next_unit = [&](int i, TileUnit &u) {
        for (i += gridDim.x; i < n_units; i += gridDim.x)
          if (tile_unit(p, i, nTB, u)) break;
        return i;
      };
      for (int i = blockIdx.x; i < n_units && ok; i += gridDim.x) {
        TileUnit u;
        if (!tile_unit(p, i, nTB, u)) {
          atomicOr(c.err, ERR_LENGTH);
          continue;
        }
        for (int j = 0; j < u.nb && ok; ++j) {
          load_block(true, true, u, j);
          if (!ok) break;
          if (j == 0) {
            load_q(i);  // of the CTA's first unit; later ones are there
            if (!ok) break;
          }
          load_block(false, false, u, j);
        }
        TileUnit v;
        const int nx = next_unit(i, v);
        if (ok && nx < n_units) load_q(nx);
        // (The last block's keys are still there.)
        for (int j = 0; j + 1 < u.nb && ok; ++j) load_block(false, true, u, j);
      }
      if (!ok) {
        if (!*abort) atomicOr(c.err, ERR_TIMEOUT);
        *abort = 1;
      }
      // Whether or not another role gave up: every load issued lands
      // (bounded) before the CTA's shared memory is given back.
      volatile int never = 0;
      for (int k = max(0, nq - 2); k < nq; ++k)
        mbar_wait_idle(smem_u32(&b_qfull[k & 1]), (uint32_t)((k / 2) & 1), &never);
      if (nk) mbar_wait_idle(smem_u32(&b_kfull), (uint32_t)((nk - 1) & 1), &never);
      if (nv) mbar_wait_idle(smem_u32(&b_vfull), (uint32_t)((nv - 1) & 1), &never);
    }
  } else if (warp == 9) {
    // Issuer (one thread's MMAs run in the order of issue; see
    // kvr_absorb_long.cu).
    int nk = 0, nv = 0, nq = 0, np = 0, nsc = 0;  // waited for; score blocks issued
    bool ok = true;
    // The candidates' new rows into their places of a staged tail block.
    auto put_new = [&](unsigned char *blk, const unsigned char *src, int t_new) {
      for (int x = lane; x < N * 16; x += 32) {
        const int row = (x >> 4) * T + t_new, ch = x & 15;
        *reinterpret_cast<int4 *>(blk + (ch >> 3) * kHalf + row * 128 +
                                  (((ch & 7) ^ (row & 7)) << 4)) =
            *reinterpret_cast<const int4 *>(src + (x >> 4) * 256 + ch * 16);
      }
      fence_proxy_async();
      __syncwarp();
    };
    // Wait for K block j, complete it.
    const unsigned char *fresh = stage;  // the unit's new rows
    auto have_k = [&](const TileUnit &u, int j) {
      if (!wait_warp(b_kfull, nk)) return false;
      ++nk;
      if (j + 1 == u.nb) put_new(smem + kTile, fresh, nt - (nTB - 1) * T);
      return true;
    };
    auto issue_s = [&](uint64_t a0, uint64_t b0, int ncol, uint64_t *freed) {
      if (lane == 0) {
        const uint32_t id = idesc_bf16(kBlk, ncol, false);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint64_t off = (uint64_t)(((k >> 2) * kHalf + (k & 3) * 32) >> 4);
          tc_mma(tm, a0 + off, b0 + off, id, k > 0);
        }
        tc_commit(smem_u32(&b_s));
        if (freed) tc_commit(smem_u32(freed));
      }
    };
    const uint64_t dQ = sdesc_sw128(aQ, 16, 1024), dK = sdesc_sw128(aK, 16, 1024),
                   dV = sdesc_sw128(aV, 16, 1024);
    for (int i = blockIdx.x; i < n_units && ok; i += gridDim.x) {
      TileUnit u;
      if (!tile_unit(p, i, nTB, u)) continue;
      const int qb = nq & 1;
      fresh = stage + qb * kNew;
      ok = wait_warp(b_qfull[qb], nq++ / 2);
      for (int j = 0; j < u.nb && ok; ++j) {
        const bool tail = j >= u.nPB;
        const int ncol = tail ? N * T : min(kBlk, (u.np - j * kBlk + 15) & ~15);
        ok = have_k(u, j);
        // The last score block's logits have been read.
        if (ok && j == 0 && nsc > 0) ok = wait_warp(b_sfree, nsc - 1);
        if (!ok) break;
        tc_fence_after();
        issue_s(dQ, dK, ncol, j + 1 < u.nb ? &b_kfree : nullptr);
        ok = wait_warp(b_vfull, nv++);
        if (!ok) break;
        unsigned char *V = smem + 2 * kTile;
        if (j + 1 == u.nb) {
          put_new(V, fresh + kMaxCand * 256, nt - (nTB - 1) * T);
        } else if (!tail && u.np - j * kBlk < ncol) {
          // V rows past the prefix, up to PV's 16-row step, meet P = 0 and
          // must be finite: zeros.
          const int v0 = u.np - j * kBlk;
          for (int x = lane; x < (ncol - v0) * 16; x += 32)
            reinterpret_cast<int4 *>(V + ((x >> 3) & 1) * kHalf + (v0 + (x >> 4)) * 128)[x & 7] =
                make_int4(0, 0, 0, 0);
          fence_proxy_async();
          __syncwarp();
        }
        ok = wait_warp(b_p, np++);
        if (!ok) break;
        tc_fence_after();
        if (lane == 0) {
          const uint32_t id = idesc_bf16(kBlk, kBlk, true);
          const uint64_t b0 = sdesc_sw128(aV, kHalf, 1024);
          for (int k = 0; k < ncol / 16; ++k) {
            const uint64_t b = b0 + (uint64_t)(k * 128);
            tc_mma_ts(tmO, tm + 16 * k, b, id, j > 0 || k > 0);
            tc_mma_ts(tmO, tm + 16 * k + 8, b, id, true);
          }
          tc_commit(smem_u32(&b_vfree));
          if (j + 1 == u.nb) tc_commit(smem_u32(&b_o));
        }
      }
      // The scores: S^T = K Q^T, first of the last block, whose keys are
      // there, then of the others.
      for (int x = 0; x < u.nb && ok; ++x) {
        if (x > 0) ok = wait_warp(b_vfull, nv++) && wait_warp(b_sfree, nsc - 1);
        if (!ok) break;
        tc_fence_after();
        issue_s(x > 0 ? dV : dK, dQ, kBlk, x > 0 ? &b_vfree : &b_kfree);
        ++nsc;
      }
      if (ok && lane == 0) tc_commit(smem_u32(&b_qfree[qb]));
    }
    __syncwarp();
    if (lane == 0) {
      if (!ok) {
        if (!*abort) atomicOr(c.err, ERR_TIMEOUT);
        *abort = 1;
      }
      // Every MMA issued has completed before TMEM is freed.
      volatile int never = 0;
      tc_commit(smem_u32(&b_drain));
      mbar_wait_idle(smem_u32(&b_drain), 0, &never);
    }
  } else {
    // Softmax: warps wq and wq + 4 share lanes 32 wq .. 32 wq + 31, candidates
    // 2 wq and 2 wq + 1; warp half hf has columns 64 hf .. 64 hf + 63.
    const int hf = warp >> 2, wq = warp & 3, r = wq * 32 + lane;
    const uint32_t lanes = (uint32_t)(wq * 32) << 16;
    const int c0 = hf * 64;
    const uint32_t tS = tm + c0 + lanes, tO = tmO + c0 + lanes;
    const int pair_bar = 1 + wq;
    float *mine = &s_x[hf][r];
    const float *theirs = &s_x[hf ^ 1][r];
    auto bar_any = [&](int id, int threads, bool x) {
      int y;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
          "barrier.cta.red.or.pred q, %2, %3, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
          : "=r"(y)
          : "r"((int)x), "r"(id), "r"(threads)
          : "memory");
      return y != 0;
    };
    // Tell the partner v; a warp whose wait ran out says so instead, and both
    // leave.
    auto exchange = [&](bool good, float v) {
      *mine = good ? v : __uint_as_float(kGaveUp);
      asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory");
      return good && __float_as_uint(*theirs) != kGaveUp;
    };
    const float scale = p.scale_log2e, inv_g = p.inv_g;
    const uint64_t scale2 = pk2(scale, scale), minus2 = pk2(-1.f, -1.f);
    int ns = 0, no = 0, nu = 0;
    bool ok = true;
    for (int i = blockIdx.x; i < n_units && ok; i += gridDim.x) {
      TileUnit u;
      if (!tile_unit(p, i, nTB, u)) continue;
      // Units alternate between the lower and the upper 16 lanes of each 32.
      const int qb = nu++ & 1, ql = lane - 16 * qb;
      const int cand = 2 * wq + (ql >= G ? 1 : 0), g = ql >= G ? ql - G : ql;
      const bool valid = ql >= 0 && ql < 2 * G && cand < N;
      const unsigned char *fresh = stage + qb * kNew;
      // For the append at the unit's end (the host launches this kernel for
      // units of equal tail length).
      int tl = nt, pos0 = 0;
      if (warp < N && lane == 0) {
        tl = f.tlen[(size_t)warp * units + u.ug];
        pos0 = c.state[4 * u.ug + 1];
      }
      float ref = 0.f, l = 0.f;
      for (int j = 0; j < u.nb; ++j) {
        const bool tail = j >= u.nPB;
        const int first = (j - u.nPB) * T;  // of a tail block: its first tail row
        const int live = min(T, nt + 1 - first);
        const int ncol = tail ? N * T : min(kBlk, u.np - j * kBlk);
        // Columns that this row sees, and that any row of the warp may.
        const int lo = tail ? cand * T : 0, hi = tail ? cand * T + live : ncol;
        const int wlo = tail ? 2 * wq * T : 0, whi = tail ? min(2 * wq + 2, N) * T : ncol;
        auto sees = [&](int k) { return c0 + 32 * k < whi && c0 + 32 * k + 32 > wlo; };
        ok = wait_warp(b_s, ns++);
        tc_fence_after();
        auto load_s = [&](int k, float(&e)[32]) {
          tmem_ld32(tS + 32 * k, e);
          tmem_wait_ld();
          if (tail || c0 + 32 * k + 32 > ncol) {
#pragma unroll
            for (int x = 0; x < 32; ++x) {
              const int col = c0 + 32 * k + x;
              e[x] = col >= lo && col < hi ? e[x] : -INFINITY;
            }
          }
        };
        float mx = -INFINITY;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (ok && sees(k)) {
            float e[32];
            load_s(k, e);
#pragma unroll
            for (int x = 0; x < 32; x += 2) mx = fmaxf(mx, fmaxf(e[x], e[x + 1]));
          }
        }
        mx *= scale;
        if (j == 0) {
          if (!exchange(ok, mx)) {
            ok = false;
            break;
          }
          mx = fmaxf(mx, *theirs);
          ref = mx == -INFINITY ? 0.f : mx;
        } else if (bar_any(pair_bar, 64, !ok || mx > ref + kLazy)) {
          if (!exchange(ok, mx)) {
            ok = false;
            break;
          }
          mx = fmaxf(mx, *theirs);
          const bool up = mx > ref + kLazy;
          // O holds the blocks before this one.
          const float fa = up ? ex2(ref - mx) : 1.f;
          if (up) ref = mx;
          l *= fa;
#pragma unroll 1
          for (int k = 0; k < 64; k += 16) {
            uint32_t o[16];
            tmem_ld16(tO + k, o);
#pragma unroll
            for (int x = 0; x < 16; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * fa);
            tmem_st16(tO + k, o);
          }
        }
        const uint64_t nref2 = pk2(-ref, -ref);
        uint64_t sum2 = pk2(0.f, 0.f);
        const int ncol16 = (ncol + 15) & ~15;  // columns that PV reads
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (sees(k)) {
            float e[32];
            load_s(k, e);
            uint32_t w[32];
#pragma unroll
            for (int x = 0; x < 32; x += 2) {
              float d0, d1;
              upk2(fma2(pk2(e[x], e[x + 1]), scale2, nref2), d0, d1);
              const uint64_t p2 = pk2(ex2(d0), ex2(d1));  // exp2(-inf) = 0 for masked keys
              sum2 = add2(sum2, p2);
              float p0, p1, r0, r1;
              upk2(p2, p0, p1);
              const uint32_t b = pack_bf16(p0, p1);
              upk2(fma2(pk2(__uint_as_float(b << 16), __uint_as_float(b & 0xFFFF0000u)),
                        minus2, p2),
                   r0, r1);
              const int at = (x >> 4) * 16 + ((x & 15) >> 1);
              w[at] = b;
              w[at + 8] = pack_bf16(r0, r1);
            }
            tmem_st32(tS + 32 * k, w);
          } else if (c0 + 32 * k < ncol16) {
            uint32_t w[32];
#pragma unroll
            for (int x = 0; x < 32; ++x) w[x] = 0u;
            tmem_st32(tS + 32 * k, w);
          }
        }
        float s0, s1;
        upk2(sum2, s0, s1);
        l += s0 + s1;
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&b_p));
      }
      if (!ok) break;
      ok = wait_warp(b_o, no);
      if (!exchange(ok, l)) {
        ok = false;
        break;
      }
      {
        l += *theirs;
        tc_fence_after();
        // The largest term is 2^(x - ref) with ref the rounded x: about 1.
        if (valid && !(l >= 0.5f && l < INFINITY)) atomicOr(c.err, ERR_NONFINITE);
        const float inv = 1.f / l;
        if (hf == 0) {
          s_norm[r] = make_float2(-ref, inv);
        }
        constexpr int osz = kOutBf16 ? 2 : 4;
        unsigned char *orow = reinterpret_cast<unsigned char *>(p.out) +
                              ((((size_t)cand * per + u.row0) * G + g) * 128 + c0) * osz;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          float o[32];
          tmem_ld32(tO + 32 * k, o);
          tmem_wait_ld();
          if (valid) {
            if (kOutBf16) {
#pragma unroll
              for (int x = 0; x < 4; ++x) {
                const float *v = o + 8 * x;
                reinterpret_cast<int4 *>(orow + 64 * k)[x] = make_int4(
                    pack_bf16(v[0] * inv, v[1] * inv), pack_bf16(v[2] * inv, v[3] * inv),
                    pack_bf16(v[4] * inv, v[5] * inv), pack_bf16(v[6] * inv, v[7] * inv));
              }
            } else {
#pragma unroll
              for (int x = 0; x < 8; ++x)
                reinterpret_cast<float4 *>(orow + 128 * k)[x] =
                    make_float4(o[4 * x] * inv, o[4 * x + 1] * inv, o[4 * x + 2] * inv,
                                o[4 * x + 3] * inv);
            }
          }
        }
      }
      // Every row's reference and sum are in place.
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&b_ref));
      // Outputs that are not finite are perhaps another candidate's doing.  (O is
      // still there: read again, off the chain that the others wait for, it
      // costs 13 us of 1,691; in the loop above 52.)
      {
        float note = 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          float o[32];
          tmem_ld32(tO + 32 * k, o);
          tmem_wait_ld();
          note += nonfinite(o);
        }
        if (valid && note != 0.f && l < INFINITY)
          outputs_alone<kOutBf16>(p, i, cand, g, c0, ref, 1.f / l);
        __syncwarp();
        tc_fence_before();
      }
      ok = wait_warp(b_ref, no++);
      for (int x = 0; x < u.nb && ok; ++x) {
        const int j = x == 0 ? u.nb - 1 : x - 1;
        const bool tail = j >= u.nPB;
        const int first = (j - u.nPB) * T, live = min(T, nt + 1 - first);
        // The scores to add to, while the contraction runs: of a prefix row
        // for the four candidates of this warp's two pairs, or of the tail
        // row of its own candidate.
        const int kc = r / T, t = r % T, row = j * kBlk + r;
        float old[4] = {0.f, 0.f, 0.f, 0.f};
        float *sc = tail ? f.tscore + ((size_t)kc * units + u.ug) * f.tstride + first + t
                         : f.pscore + ((size_t)(4 * hf) * units + u.ug) * c.sstride + row;
        const size_t step = units * c.sstride;  // to the next candidate's
        const bool mine_t = tail && hf == 0 && r < N * T && t < live;
        if (mine_t && first + t != nt) old[0] = *sc;  // (the appended row starts at zero)
        if (!tail && row < u.np) {
#pragma unroll
          for (int y = 0; y < 4; ++y)
            if (4 * hf + y < N) old[y] = sc[y * step];
        }
        ok = wait_warp(b_s, ns++);
        if (!ok) break;
        tc_fence_after();
        // Head sums of this thread's key for the two candidates of pair pr.
        auto sums = [&](int pr, float &even, float &odd) {
          float e[16];
          const int at = 32 * pr + 16 * qb;
          tmem_ld16f_nowait(tm + lanes + at, e);
          tmem_wait_ld();
          const float4 *nm = reinterpret_cast<const float4 *>(&s_norm[at]);
          even = odd = 0.f;
#pragma unroll
          for (int x = 0; x < 16; x += 2) {
            const float4 z = nm[x >> 1];
            const float v0 = ex2(fmaf(e[x], scale, z.x)) * z.y;
            const float v1 = ex2(fmaf(e[x + 1], scale, z.z)) * z.w;
            if (x < G) even += v0;
            else if (x < 2 * G) odd += v0;
            if (x + 1 < G) even += v1;
            else if (x + 1 < 2 * G) odd += v1;
          }
        };
        if (!tail) {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            if (4 * hf + 2 * q < N) {
              float a, b;
              sums(2 * hf + q, a, b);
              if (row < u.np) {
                sc[2 * q * step] = old[2 * q] + a * inv_g;
                if (4 * hf + 2 * q + 1 < N) sc[(2 * q + 1) * step] = old[2 * q + 1] + b * inv_g;
              }
            }
          }
        } else if (hf == 0 && 32 * wq < N * T) {
          float a, b;
          sums((32 * wq / T) >> 1, a, b);
          if (mine_t) *sc = old[0] + ((kc & 1) ? b : a) * inv_g;
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&b_sfree));
      }
      // The pair leaves together, or not at all (its barrier counts on both).
      if (bar_any(pair_bar, 64, !ok)) {
        ok = false;
        break;
      }
      // The append: one warp a candidate, from the staged rows.
      if (warp < N) {
        const size_t cu = (size_t)warp * units + u.ug;
        __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(lane < 16 ? f.TK : f.TV) +
                             (cu * (size_t)f.tcap + nt) * 128;
        reinterpret_cast<int4 *>(dst)[lane & 15] = *reinterpret_cast<const int4 *>(
            fresh + ((lane < 16 ? 0 : kMaxCand) + warp) * 256 + (lane & 15) * 16);
        if (lane == 0) {
          if (tl != nt) atomicOr(c.err, ERR_LENGTH);
          f.tpos[cu * f.tstride + nt] = pos0 + nt;
          f.tlen[cu] = nt + 1;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&b_qfree[qb]));
    }
    if (!ok && lane == 0) {
      if (!*abort) atomicOr(c.err, ERR_TIMEOUT);
      *abort = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) tmem_dealloc(tm, kCols);
}

}  // namespace

int fork_tile_max_cand() { return kMaxCand; }
int fork_tile_box_rows() { return kBox; }
int fork_tile_tail_rows(int n_cand) {
  return n_cand >= 1 && n_cand <= kMaxCand ? tail_rows(n_cand) : 0;
}

cudaError_t launch_fork_tile(const CUtensorMap &tmK, const CUtensorMap &tmV,
                             const CUtensorMap &tmTK, const CUtensorMap &tmTV,
                             const CUtensorMap &tmQ, const ForkTileParams &p, int sms,
                             cudaStream_t st) {
  if (p.f.N < 1 || p.f.N > kMaxCand || p.f.p.G > 8 || p.nt < 0 || p.nt + 1 > p.f.tcap)
    return cudaErrorInvalidValue;
  const int units = p.f.p.S * p.nl * p.f.p.H;
  auto kern = p.f.p.out_bf16 ? fork_tile_kernel<true> : fork_tile_kernel<false>;
  cudaError_t e =
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(units < 2 * sms ? units : 2 * sms), dim3(kThr), (size_t)kSmem, st,
                    p, tmK, tmV, tmTK, tmTV, tmQ, units);
}

}  // namespace kvr
