// kvr_absorb_long.cu -- absorbing a chunk of tokens into units of any length
// (bf16 in and out, head_dim 128, G <= 8): what kvr_absorb_chunk runs beyond
// the limits of the one-launch kernels of kvr_absorb.cu, a prompt's prefill
// among it (Algorithm 1: one forward pass over an accepted step, or over the
// prompt; Sec. 2.1: every token adds its head-mean probabilities to the
// scores of the rows it attends; then one eviction).
//
// The work is a contraction: C tokens x G heads against m + C rows, causal.
// Run token by token it was one launch a token, each reading every row again
// (7B, two 1,000-token prompts: 140 ms; 16 sequences absorbing 57 tokens into
// 640 rows: 39.8 ms).  Here it is four steps (0.90 ms and 0.73 ms):
//   1. append: the chunk's rows go to slots m.. of each unit, score 0.
//   2. attend (tcgen05): tiles of 128 query rows (128 / G whole tokens) over
//      128-row key blocks with an online softmax; writes the outputs and each
//      query row's log2 normaliser (into the cache's logit scratch).
//   3. score (tcgen05): S^T = K Q^T, keys on the lanes, so a key's column sum
//      over all queries is a sum inside one thread; the probabilities come
//      exactly from the normalisers, and each key's sum is added once.
//   4. finish: lengths, and the eviction where one is due (kvr_generic.cu).
// Sums in another order can trade two rows whose scores agree to their
// rounding, and the freed slots are filled in order, so that one traded row
// moves others: where the rows around the cut lie that close, their scores are
// formed again token by token, by the generic kernel's arithmetic to the bit,
// and the rows that stay are those that a token-by-token absorb of the same
// state keeps (kvr_generic.cu).
// Recomputing Q K^T in 3 costs one contraction of four, against column sums
// over the lanes in 2 (124 shuffles a warp and block) and probabilities that
// are only final after a row's last block.
//
// Precision: Q K^T accumulates in fp32; P is split into two bf16 terms (hi +
// lo, 16 bits of mantissa) for PV, as in kvr_absorb.cu; outputs are bf16.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include "kvr_internal.h"
#include "kvr_tmem.cuh"

namespace kvr {
namespace {

using namespace ptx;

constexpr int kBlk = 128;            // keys a block; query rows a tile
constexpr int kHalf = kBlk * 128;    // bytes of a 64-column half of a block
constexpr int kTile = 2 * kHalf;     // bytes of a 128 x 128 bf16 block
constexpr int kBox = 32;             // slab rows a TMA box
constexpr int kAttThr = 320, kAttCols = 256;  // attend: two CTAs an SM
constexpr int kAttSmem = 3 * kTile + 1024;
static_assert(kAttSmem + 2048 <= 113 * 1024, "two CTAs an SM, with the static variables");
// Score: one CTA an SM; four softmax warpgroups, a loading and an issuing warp.
constexpr int kScThr = 576, kScCols = 512;
constexpr int kProducer = 16, kIssuer = 17;
constexpr int kQRing = 3;            // query tiles in flight
constexpr int kLRing = 4;            // their rows' normalisers
struct ScoreBars {
  uint64_t kfull[2], kfree[2], qfull[kQRing], qfree[kQRing], lfull[kLRing], lfree[kLRing],
      s[2][2], sfree[2][2], drain;
  uint32_t tmem;
  int abort;
};
constexpr int kScoreSmem = (4 + kQRing) * kTile + kLRing * 512 + (int)sizeof(ScoreBars);
static_assert(kScoreSmem <= 227 * 1024, "one CTA an SM");
// Lazy rescaling: the reference of a row's exponentials moves only when a
// logit exceeds it by 2^kLazy; sums stay far inside fp32's range.
constexpr float kLazy = 8.f;
constexpr uint32_t kGaveUp = 0x7FBADBADu;  // a NaN that no arithmetic returns

// The unit of index x in [0, S * nl * H) and the first token row of its
// (sequence, layer) in q, k_new, v_new and out.
struct LUnit {
  size_t ug, row0;
  int h, m;  // m: rows before the chunk
};
__device__ __forceinline__ LUnit unit_at(const AbsorbParams &p, int x) {
  const CacheView &c = p.c;
  LUnit u;
  u.h = x % c.H;
  u.ug = unit_index(c, p.lb, p.nl, x);
  u.row0 = (size_t)(x / c.H) * p.chunk;
  u.m = c.state[4 * u.ug];
  return u;
}
// Rows the unit could not hold: the host checked its mirror, so this says
// that the device lengths are not what the host thinks; such units are left
// alone by every kernel below.
__device__ __forceinline__ bool unit_ok(const AbsorbParams &p, const LUnit &u) {
  return u.m >= 0 && u.m + p.chunk <= p.c.cap && u.m + p.chunk <= p.max_rows;
}

// ---- 1. append ----------------------------------------------------------------

constexpr int kAppendRows = 32;    // rows a CTA copies at a time
constexpr int kAppendCtas = 1024;  // CTAs a unit, at most

__global__ void __launch_bounds__(256) long_append_kernel(const AbsorbParams p) {
  pdl_begin();
  const CacheView &c = p.c;
  const LUnit u = unit_at(p, blockIdx.x);
  if (p.settle && blockIdx.y == 0 && threadIdx.x == 0) {
    c.state[4 * u.ug + 2] = 0;  // the key sum's place is the ties' now
    if (blockIdx.x == 0) tie_words(c, u.ug)[kTieUnits] = 0;
  }
  if (!unit_ok(p, u)) {
    if (threadIdx.x == 0)
      atomicOr(c.err, u.m >= 0 && u.m + p.chunk > c.cap ? ERR_CAPACITY : ERR_LENGTH);
    return;
  }
  const int4 *kn = reinterpret_cast<const int4 *>(p.k_new);
  const int4 *vn = reinterpret_cast<const int4 *>(p.v_new);
  const int next = c.state[4 * u.ug + 1];
  for (int j0 = blockIdx.y * kAppendRows; j0 < p.chunk; j0 += gridDim.y * kAppendRows) {
    const int nr = min(kAppendRows, p.chunk - j0);
    const size_t dst = u.ug * (size_t)c.cap + u.m + j0;
    int4 *K = reinterpret_cast<int4 *>(c.K) + dst * 16;
    int4 *V = reinterpret_cast<int4 *>(c.V) + dst * 16;
    for (int i = threadIdx.x; i < nr * 16; i += 256) {
      const size_t src = ((u.row0 + j0 + (i >> 4)) * c.H + u.h) * 16 + (i & 15);
      const int4 a = kn[src], b = vn[src];
      K[i] = a;
      V[i] = b;
    }
    if ((int)threadIdx.x < nr) {
      const size_t s = u.ug * (size_t)c.sstride + u.m + j0 + threadIdx.x;
      c.score[s] = 0.f;
      c.pos[s] = next + j0 + (int)threadIdx.x;
    }
  }
}

// ---- 2. attend ----------------------------------------------------------------

// One work item: a query tile (128 / G whole tokens) of one unit.
struct AttItem {
  LUnit u;
  int tok0, toks;  // first token; tokens
  int lim, nb;     // rows the last token sees; key blocks
};

__device__ __forceinline__ bool att_item(const AbsorbParams &p, int i, int units, int n_qt,
                                         int Jt, AttItem &it) {
  // The longest tiles (the last tokens) of every unit first.
  const int tile = n_qt - 1 - i / units;
  it.u = unit_at(p, i % units);
  it.tok0 = tile * Jt;
  it.toks = min(Jt, p.chunk - it.tok0);
  it.lim = it.u.m + it.tok0 + it.toks;
  it.nb = (it.lim + kBlk - 1) / kBlk;
  return unit_ok(p, it.u);
}

// Two CTAs an SM, each with one tile: while one waits for its loads, its
// softmax or its outputs, the other has the tensor cores.  7B, two 1,000-token
// prompts: 0.58 ms, against 0.80 ms for one CTA with two tiles in step that
// share the K and V blocks (a third of it passed between items) and 0.94 ms
// for that with one softmax warp for 32 rows instead of two.  Eight softmax
// warps, then a loading and an issuing warp.
__global__ void __launch_bounds__(kAttThr, 2)
    long_attend_kernel(const AbsorbParams p, const __grid_constant__ CUtensorMap tmK,
                       const __grid_constant__ CUtensorMap tmV,
                       const __grid_constant__ CUtensorMap tmQ, float *lse, int n_items,
                       int n_qt, int out32) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  __shared__ float s_x[2][kBlk];  // what a row's two threads tell each other
  __shared__ __align__(8) uint64_t b_qfull, b_qfree, b_kfull, b_kfree, b_vfull, b_vfree, b_s,
      b_p, b_o, b_drain;
  unsigned char *smem = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const uint32_t aQ = smem_u32(smem), aK = aQ + kTile, aV = aK + kTile;
  const CacheView &c = p.c;
  const int G = c.G, Jt = kBlk / G, units = n_items / n_qt;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  volatile int *abort = &s_abort;
  // A whole warp's bounded wait; its lanes agree on the result.
  auto wait_warp = [&](uint64_t &bar, int n) {
    return __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar), (uint32_t)(n & 1), abort)) != 0;
  };
  if (warp == 8) tmem_alloc(smem_u32(&s_tmem), kAttCols);
  if (tid == 0) {
    mbar_init(smem_u32(&b_qfull), 1);
    mbar_init(smem_u32(&b_qfree), 1);
    mbar_init(smem_u32(&b_kfull), 1);
    mbar_init(smem_u32(&b_kfree), 1);
    mbar_init(smem_u32(&b_vfull), 1);
    mbar_init(smem_u32(&b_vfree), 1);
    mbar_init(smem_u32(&b_s), 1);
    mbar_init(smem_u32(&b_p), 8);
    mbar_init(smem_u32(&b_o), 1);
    mbar_init(smem_u32(&b_drain), 1);
    s_abort = 0;
    fence_mbar_init();
  }
  // Query rows past the whole tokens of a tile are never loaded: zeros.
  for (int i = tid; i < 2 * (kBlk - Jt * G) * 8; i += kAttThr) {
    const int row = Jt * G + (i >> 3) % (kBlk - Jt * G), hf = (i >> 3) / (kBlk - Jt * G);
    reinterpret_cast<int4 *>(smem + hf * kHalf + row * 128)[i & 7] = make_int4(0, 0, 0, 0);
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  const uint32_t tm = s_tmem, tmO = tm + kBlk;

  if (warp == 8) {
    // Producer: one thread issues every load, in the order they are used.
    if (lane == 0) {
      prefetch_tmap(&tmK);
      prefetch_tmap(&tmV);
      prefetch_tmap(&tmQ);
      const uint32_t q_bytes = 256u * (uint32_t)(G * Jt);
      int nq = 0, nkv = 0;  // query tiles and blocks issued
      bool ok = true;
      auto load_block = [&](const CUtensorMap *map, uint32_t dst, uint64_t &full,
                            uint64_t &freed, int row, int rows) {
        if (ok && nkv > 0) ok = mbar_wait(smem_u32(&freed), (uint32_t)((nkv - 1) & 1), abort);
        if (!ok) return;
        const int nbox = (rows + kBox - 1) / kBox;
        const uint32_t bar = smem_u32(&full);
        mbar_expect_tx(bar, (uint32_t)nbox * 2 * kBox * 128);
        for (int b = 0; b < nbox; ++b)
          for (int hf = 0; hf < 2; ++hf)
            tma_load_2d(dst + hf * kHalf + b * kBox * 128, map, 64 * hf, row + b * kBox, bar);
      };
      int nk = 0, nv = 0;  // loads in flight to wait for at the end
      for (int i = blockIdx.x; i < n_items && ok; i += gridDim.x) {
        AttItem it;
        if (!att_item(p, i, units, n_qt, Jt, it)) continue;
        const int row0 = (int)(it.u.ug * (size_t)c.cap);
        for (int j = 0; j < it.nb && ok; ++j) {
          const int rows = min(kBlk, it.lim - j * kBlk);
          load_block(&tmK, aK, b_kfull, b_kfree, row0 + j * kBlk, rows);
          if (!ok) break;
          ++nk;
          if (j == 0) {
            if (nq > 0) ok = mbar_wait(smem_u32(&b_qfree), (uint32_t)((nq - 1) & 1), abort);
            if (!ok) break;
            mbar_expect_tx(smem_u32(&b_qfull), q_bytes);
            for (int hf = 0; hf < 2; ++hf)
              tma_load_4d(aQ + hf * kHalf, &tmQ, 64 * hf, 0, it.u.h, (int)it.u.row0 + it.tok0,
                          smem_u32(&b_qfull));
            ++nq;
          }
          load_block(&tmV, aV, b_vfull, b_vfree, row0 + j * kBlk, rows);
          if (!ok) break;
          ++nv;
          ++nkv;
        }
      }
      if (!ok) {
        if (!*abort) atomicOr(c.err, ERR_TIMEOUT);
        *abort = 1;
      }
      // Whether or not another role gave up: every load issued lands
      // (bounded) before the CTA's shared memory is given back.
      volatile int never = 0;
      if (nq) mbar_wait(smem_u32(&b_qfull), (uint32_t)((nq - 1) & 1), &never);
      if (nk) mbar_wait(smem_u32(&b_kfull), (uint32_t)((nk - 1) & 1), &never);
      if (nv) mbar_wait(smem_u32(&b_vfull), (uint32_t)((nv - 1) & 1), &never);
    }
  } else if (warp == 9) {
    // Issuer: S(j) = Q K_j^T, then O += P(j) V_j once the softmax has put P
    // in place of S.  One thread issues, and its MMAs run in the order of
    // issue, so S(j + 1) may follow PV(j), whose P it replaces.
    int nk = 0, nv = 0, nq = 0;
    bool ok = true;
    for (int i = blockIdx.x; i < n_items && ok; i += gridDim.x) {
      AttItem it;
      if (!att_item(p, i, units, n_qt, Jt, it)) continue;
      for (int j = 0; j < it.nb; ++j) {
        const int ncol = min(kBlk, (it.lim - j * kBlk + 15) & ~15);
        ok = wait_warp(b_kfull, nk++) && (j > 0 || wait_warp(b_qfull, nq++));
        if (!ok) break;
        tc_fence_after();
        if (lane == 0) {
          const uint32_t id = idesc_bf16(kBlk, ncol, false);
          const uint64_t a0 = sdesc_sw128(aQ, 16, 1024), b0 = sdesc_sw128(aK, 16, 1024);
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint64_t off = (uint64_t)(((k >> 2) * kHalf + (k & 3) * 32) >> 4);
            tc_mma(tm, a0 + off, b0 + off, id, k > 0);
          }
          tc_commit(smem_u32(&b_s));
          tc_commit(smem_u32(&b_kfree));
          if (j + 1 == it.nb) tc_commit(smem_u32(&b_qfree));
        }
        ok = wait_warp(b_vfull, nv);
        if (!ok) break;
        // V rows past the last one that the tile sees, up to the 16-row step of
        // PV, meet P = 0 and must be finite: zeros.  (They are a later tile's,
        // or the cache's slots past the unit's end, which may hold anything.)
        const int v0 = it.lim - j * kBlk;
        if (v0 < ncol) {
          unsigned char *V = smem + 2 * kTile;
          for (int x = lane; x < (ncol - v0) * 16; x += 32)
            reinterpret_cast<int4 *>(V + ((x >> 3) & 1) * kHalf + (v0 + (x >> 4)) * 128)[x & 7] =
                make_int4(0, 0, 0, 0);
          fence_proxy_async();
          __syncwarp();
        }
        ok = wait_warp(b_p, nv++);
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
          if (j + 1 == it.nb) tc_commit(smem_u32(&b_o));
        }
      }
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
      mbar_wait(smem_u32(&b_drain), 0, &never);
    }
  } else {
    // Softmax: two warpgroups, each with half of a block's columns; thread r
    // of either owns query row r.  The warps of the two that share 32 rows
    // agree on the rows' reference over a named barrier.
    const int hf = warp >> 2, wq = warp & 3, r = wq * 32 + lane;
    const uint32_t lanes = (uint32_t)(wq * 32) << 16;
    const int c0 = hf * 64;
    const uint32_t tS = tm + c0 + lanes, tO = tmO + c0 + lanes;
    const int pair_bar = 1 + wq;
    float *mine = &s_x[hf][r];
    const float *theirs = &s_x[hf ^ 1][r];
    auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(pair_bar) : "memory"); };
    auto pair_any = [&](bool x) {
      int y;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
          "barrier.cta.red.or.pred q, %2, 64, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
          : "=r"(y)
          : "r"((int)x), "r"(pair_bar)
          : "memory");
      return y != 0;
    };
    // Tell the partner v; a warp whose wait ran out says so instead, and both
    // leave (no warp is left at the pair's barrier).
    auto exchange = [&](bool good, float v) {
      *mine = good ? v : __uint_as_float(kGaveUp);
      pair_sync();
      return good && __float_as_uint(*theirs) != kGaveUp;
    };
    const float scale = p.scale_log2e;
    const uint64_t scale2 = pk2(scale, scale), minus2 = pk2(-1.f, -1.f);
    const int tk = r / G;
    int ns = 0, no = 0;
    bool ok = true;
    for (int i = blockIdx.x; i < n_items && ok; i += gridDim.x) {
      AttItem it;
      if (!att_item(p, i, units, n_qt, Jt, it)) continue;
      const bool valid = tk < it.toks && r < Jt * G;
      // Rows the query sees (rows past the tile's tokens follow the last),
      // and the first query of this warp; of this half's columns.
      const int first = it.u.m + it.tok0 + 1 - c0;
      const int seen = first + min(tk, it.toks - 1);
      const int seen_w = first + min(32 * wq / G, it.toks - 1);
      float ref = 0.f, l = 0.f;
      for (int j = 0; j < it.nb; ++j) {
        ok = wait_warp(b_s, ns++);
        tc_fence_after();
        // This half's columns in use, 32 at a time: a first reading for the
        // maximum, a second for the exponentials (TMEM reads are cheap; the
        // registers to keep 64 logits are not there).
        const int ncol = it.lim - c0 - j * kBlk, lim = seen - j * kBlk,
                  lim_w = seen_w - j * kBlk;
        auto load_s = [&](int k, float(&e)[32]) {
          tmem_ld32(tS + 32 * k, e);
          tmem_wait_ld();
          if (lim_w < 32 * k + 32) {
#pragma unroll
            for (int x = 0; x < 32; ++x) e[x] = 32 * k + x < lim ? e[x] : -INFINITY;
          }
        };
        float mx = -INFINITY;
        if (ok && lim_w >= 64) {  // every column is seen: both loads in flight
          float e0[32], e1[32];
          tmem_ld32(tS, e0);
          tmem_ld32(tS + 32, e1);
          tmem_wait_ld();
#pragma unroll
          for (int x = 0; x < 32; ++x) mx = fmaxf(mx, fmaxf(e0[x], e1[x]));
        } else {
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            if (ok && 32 * k < ncol) {
              float e[32];
              load_s(k, e);
#pragma unroll
              for (int x = 0; x < 32; x += 2) mx = fmaxf(mx, fmaxf(e[x], e[x + 1]));
            }
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
        } else if (pair_any(!ok || mx > ref + kLazy)) {
          if (!exchange(ok, mx)) {
            ok = false;
            break;
          }
          mx = fmaxf(mx, *theirs);
          const bool up = mx > ref + kLazy;
          // O holds the blocks before this one (S of this block was
          // committed after their PV).
          const float f = up ? ex2(ref - mx) : 1.f;
          if (up) ref = mx;
          l *= f;
#pragma unroll 1
          for (int k = 0; k < 64; k += 16) {
            uint32_t o[16];
            tmem_ld16(tO + k, o);
#pragma unroll
            for (int x = 0; x < 16; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * f);
            tmem_st16(tO + k, o);
          }
        }
        const uint64_t nref2 = pk2(-ref, -ref);
        uint64_t sum2 = pk2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (32 * k < ncol) {
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
              // p - bf16(p), exact
              upk2(fma2(pk2(__uint_as_float(b << 16), __uint_as_float(b & 0xFFFF0000u)),
                        minus2, p2),
                   r0, r1);
              const int at = (x >> 4) * 16 + ((x & 15) >> 1);
              w[at] = b;
              w[at + 8] = pack_bf16(r0, r1);
            }
            tmem_st32(tS + 32 * k, w);  // 8 hi then 8 lo columns each 16 keys
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
      ok = wait_warp(b_o, no++);
      if (!exchange(ok, l)) {
        ok = false;
        break;
      }
      l += *theirs;
      tc_fence_after();
      // The largest term is 2^(x - ref) with ref the rounded x: about 1.
      if (valid && !(l >= 0.5f && l < INFINITY)) atomicOr(c.err, ERR_NONFINITE);
      const float inv = 1.f / l;
      const size_t qrow = ((it.u.row0 + it.tok0 + tk) * c.H + it.u.h) * G + (r - tk * G);
      unsigned char *orow = reinterpret_cast<unsigned char *>(p.out) + qrow * 256 + 128 * hf;
      float note = 0.f;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        float o[32];
        tmem_ld32(tO + 32 * k, o);
        tmem_wait_ld();
        note += nonfinite(o);
        if (valid) {
          uint32_t w[16];
#pragma unroll
          for (int x = 0; x < 16; ++x) w[x] = pack_bf16(o[2 * x] * inv, o[2 * x + 1] * inv);
          if (out32) {
            st_global32(orow + 64 * k, w);
            st_global32(orow + 64 * k + 32, w + 8);
          } else {
#pragma unroll
            for (int x = 0; x < 4; ++x)
              reinterpret_cast<int4 *>(orow + 64 * k)[x] =
                  make_int4(w[4 * x], w[4 * x + 1], w[4 * x + 2], w[4 * x + 3]);
          }
        }
      }
      if (valid && note != 0.f && l < INFINITY) {
        // Perhaps not this row's doing: its outputs from the rows it sees.
        const size_t row = it.u.ug * (size_t)c.cap * 128;
        for (int k = 0; k < 2; ++k) {
          float o[32];
          for (int x = 0; x < 32; ++x) o[x] = 0.f;
          attend_row(p.q + qrow * 128, reinterpret_cast<const __nv_bfloat16 *>(c.K) + row,
                     reinterpret_cast<const __nv_bfloat16 *>(c.V) + row,
                     it.u.m + it.tok0 + tk + 1, c0 + 32 * k, scale, ref, o);
          for (int x = 0; x < 16; ++x)
            reinterpret_cast<uint32_t *>(orow + 64 * k)[x] =
                pack_bf16(o[2 * x] * inv, o[2 * x + 1] * inv);
        }
      }
      __syncwarp();
      if (valid && hf == 0)
        lse[it.u.ug * (size_t)G * c.cap + (size_t)it.tok0 * G + r] = ref + log2f(l);
      tc_fence_before();
      pair_sync();  // the partner has read this row's sum
    }
    if (!ok && lane == 0) {
      if (!*abort) atomicOr(c.err, ERR_TIMEOUT);
      *abort = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) tmem_dealloc(tm, kAttCols);
}

// ---- 3. score -----------------------------------------------------------------

// One work item: 256 rows (two key tiles) of one unit, against every query
// tile that sees one of them.
struct ScoreItem {
  LUnit u;
  int k0, n, Jt;  // first row; rows of the unit; tokens a query tile
  // Of key tile t: the first query tile that sees one of its rows, and its
  // rows (<= 0: none).
  __device__ int q0(int t) const { return max(0, k0 + t * kBlk - u.m) / Jt; }
  __device__ int nk(int t) const { return min(kBlk, n - k0 - t * kBlk); }
};

__device__ __forceinline__ bool score_item(const AbsorbParams &p, int i, int Jt,
                                           ScoreItem &it) {
  // The first rows, which every token sees, of every unit first.
  const int units = p.c.S * p.nl * p.c.H, kp = i / units;
  it.u = unit_at(p, i % units);
  if (!unit_ok(p, it.u)) return false;
  it.n = it.u.m + p.chunk;
  it.k0 = 2 * kBlk * kp;
  it.Jt = Jt;
  return it.k0 < it.n;
}

__global__ void __launch_bounds__(kScThr, 1)
    long_score_kernel(const AbsorbParams p, const __grid_constant__ CUtensorMap tmK,
                      const __grid_constant__ CUtensorMap tmQ, const float *lse, int n_items,
                      int n_qt) {
  // (No static shared memory: the tiles need 1,024-byte alignment and all the
  // rest of the SM's shared memory.)
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t aK = smem_u32(smem), aQ = aK + 4 * kTile;
  float *s_lse = reinterpret_cast<float *>(smem + (4 + kQRing) * kTile);  // [kLRing][128]
  ScoreBars &B = *reinterpret_cast<ScoreBars *>(s_lse + kLRing * kBlk);
  const CacheView &c = p.c;
  const int G = c.G, Jt = kBlk / G;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  volatile int *abort = &B.abort;
  // A whole warp's bounded wait for completion n of a barrier.
  auto wait_warp = [&](uint64_t &bar, int n) {
    return __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar), (uint32_t)(n & 1), abort)) != 0;
  };
  if (warp == kProducer) tmem_alloc(smem_u32(&B.tmem), kScCols);
  if (tid == 0) {
    for (int t = 0; t < 2; ++t) {
      mbar_init(smem_u32(&B.kfull[t]), 1);
      mbar_init(smem_u32(&B.kfree[t]), 1);
      for (int b = 0; b < 2; ++b) {
        mbar_init(smem_u32(&B.s[t][b]), 1);
        mbar_init(smem_u32(&B.sfree[t][b]), 4);
      }
    }
    for (int s = 0; s < kQRing; ++s) {
      mbar_init(smem_u32(&B.qfull[s]), 1);
      mbar_init(smem_u32(&B.qfree[s]), 1);
    }
    for (int s = 0; s < kLRing; ++s) {
      mbar_init(smem_u32(&B.lfull[s]), 32);
      mbar_init(smem_u32(&B.lfree[s]), 8);
    }
    mbar_init(smem_u32(&B.drain), 1);
    B.abort = 0;
    fence_mbar_init();
  }
  for (int i = tid; i < kQRing * 2 * (kBlk - Jt * G) * 8; i += kScThr) {
    const int row = Jt * G + (i >> 3) % (kBlk - Jt * G), hf = (i >> 3) / (kBlk - Jt * G);
    reinterpret_cast<int4 *>(smem + 4 * kTile + hf * kHalf + row * 128)[i & 7] =
        make_int4(0, 0, 0, 0);
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_begin();
  const uint32_t tm = B.tmem;

  if (warp == kProducer) {
    // Producer: key tiles (two pairs in flight), query tiles and their
    // rows' normalisers.
    if (lane == 0) {
      prefetch_tmap(&tmK);
      prefetch_tmap(&tmQ);
    }
    const uint32_t q_bytes = 256u * (uint32_t)(G * Jt);
    int nk = 0, nq = 0;
    bool ok = true;
    for (int i = blockIdx.x; i < n_items && ok; i += gridDim.x) {
      ScoreItem it;
      if (!score_item(p, i, Jt, it)) continue;
      const int kb = nk & 1;
      if (nk >= 2) ok = wait_warp(B.kfree[kb], nk / 2 - 1);
      if (!ok) break;
      if (lane == 0) {
        const int rows = min(2 * kBlk, it.n - it.k0), nbox = (rows + kBox - 1) / kBox;
        const uint32_t bar = smem_u32(&B.kfull[kb]);
        const int row = (int)(it.u.ug * (size_t)c.cap) + it.k0;
        mbar_expect_tx(bar, (uint32_t)nbox * 2 * kBox * 128);
        for (int b = 0; b < nbox; ++b)
          for (int hf = 0; hf < 2; ++hf)
            tma_load_2d(aK + (kb * 2 + b / 4) * kTile + hf * kHalf + (b & 3) * kBox * 128, &tmK,
                        64 * hf, row + b * kBox, bar);
      }
      ++nk;
      const float *lu = lse + it.u.ug * (size_t)G * c.cap;
      for (int q = it.q0(0); q < n_qt; ++q) {
        const int s = nq % kQRing;
        const int base = q * Jt * G, nv = min(Jt, p.chunk - q * Jt) * G;
        float v[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int col = 32 * x + lane;
          v[x] = col < nv ? lu[base + col] : INFINITY;
        }
        if (nq >= kQRing) ok = wait_warp(B.qfree[s], nq / kQRing - 1);
        if (!ok) break;
        if (lane == 0) {
          const uint32_t bar = smem_u32(&B.qfull[s]);
          mbar_expect_tx(bar, q_bytes);
          for (int hf = 0; hf < 2; ++hf)
            tma_load_4d(aQ + s * kTile + hf * kHalf, &tmQ, 64 * hf, 0, it.u.h,
                        (int)it.u.row0 + q * Jt, bar);
        }
        // The normalisers have slots of their own: the softmax still reads
        // them when the contraction has long released the query tile.  (In
        // one slot with it, the three query tiles in flight waited for the
        // softmax: 249 us against 227, 7B, two 1,000-token prompts.)
        const int sl = nq % kLRing;
        ++nq;
        if (nq > kLRing) ok = wait_warp(B.lfree[sl], (nq - 1) / kLRing - 1);
        if (!ok) break;
#pragma unroll
        for (int x = 0; x < 4; ++x) s_lse[sl * kBlk + 32 * x + lane] = -v[x];
        mbar_arrive(smem_u32(&B.lfull[sl]));
      }
    }
    __syncwarp();
    if (lane == 0) {
      if (!ok) {
        if (!*abort) atomicOr(c.err, ERR_TIMEOUT);
        *abort = 1;
      }
      volatile int never = 0;
      for (int k = max(0, nk - 2); k < nk; ++k)
        mbar_wait(smem_u32(&B.kfull[k & 1]), (uint32_t)((k / 2) & 1), &never);
      for (int k = max(0, nq - kQRing); k < nq; ++k)
        mbar_wait(smem_u32(&B.qfull[k % kQRing]), (uint32_t)((k / kQRing) & 1), &never);
    }
  } else if (warp == kIssuer) {
    int nk = 0, nq = 0, ns0 = 0, ns1 = 0;
    bool ok = true;
    const uint32_t id = idesc_bf16(kBlk, kBlk, false);
    for (int i = blockIdx.x; i < n_items && ok; i += gridDim.x) {
      ScoreItem it;
      if (!score_item(p, i, Jt, it)) continue;
      const int kb = nk & 1;
      ok = wait_warp(B.kfull[kb], nk / 2);
      for (int q = it.q0(0); q < n_qt && ok; ++q) {
        const int s = nq % kQRing;
        ok = wait_warp(B.qfull[s], nq / kQRing);
        for (int t = 0; t < 2 && ok; ++t) {
          if (it.nk(t) <= 0 || q < it.q0(t)) continue;
          int &ns = t ? ns1 : ns0;
          const int b = ns & 1;
          if (ns >= 2) ok = wait_warp(B.sfree[t][b], ns / 2 - 1);
          if (!ok) break;
          ++ns;
          tc_fence_after();
          if (lane == 0) {
            const uint64_t a0 = sdesc_sw128(aK + (kb * 2 + t) * kTile, 16, 1024);
            const uint64_t b0 = sdesc_sw128(aQ + s * kTile, 16, 1024);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const uint64_t off = (uint64_t)(((k >> 2) * kHalf + (k & 3) * 32) >> 4);
              tc_mma(tm + (t * 2 + b) * kBlk, a0 + off, b0 + off, id, k > 0);
            }
            tc_commit(smem_u32(&B.s[t][b]));
          }
        }
        if (!ok) break;
        if (lane == 0) tc_commit(smem_u32(&B.qfree[s]));
        ++nq;
      }
      if (!ok) break;
      if (lane == 0) tc_commit(smem_u32(&B.kfree[kb]));
      ++nk;
    }
    if (lane == 0) {
      if (!ok) {
        if (!*abort) atomicOr(c.err, ERR_TIMEOUT);
        *abort = 1;
      }
      volatile int never = 0;
      tc_commit(smem_u32(&B.drain));
      mbar_wait(smem_u32(&B.drain), 0, &never);
    }
  } else if (warp < kProducer) {
    // Two warpgroups a key tile, which take its S buffers in turn; thread r
    // of either owns key row r.
    const int t = warp >> 3, b = (warp >> 2) & 1, wq = warp & 3, r = wq * 32 + lane;
    const uint32_t tS = tm + (t * 2 + b) * kBlk + ((uint32_t)(wq * 32) << 16);
    const uint64_t scale2 = pk2(p.scale_log2e, p.scale_log2e);
    int nq = 0, ns = 0;
    bool ok = true;
    for (int i = blockIdx.x; i < n_items && ok; i += gridDim.x) {
      ScoreItem it;
      if (!score_item(p, i, Jt, it)) continue;
      const int slot = it.k0 + t * kBlk + r;
      const int tmin = max(0, slot - it.u.m);  // first token that sees the row
      const int tmin_w = max(0, it.k0 + t * kBlk + wq * 32 + 31 - it.u.m);
      const int q1 = it.nk(t) > 0 ? it.q0(t) : n_qt;
      // The row's sum: of each query tile's 128 terms apart, then over the
      // tiles.  (What is left of the scores' error, about 1.2e-7 relative, is the
      // contraction's accumulation: compensated sums did not move it.)
      float sum = 0.f;
      for (int q = it.q0(0); q < n_qt; ++q) {
        const int s = nq % kLRing, ph_l = nq / kLRing;
        ++nq;
        // One of the tile's two warpgroups releases each tile's normalisers: the one
        // that reads it, or the first where the tile has nothing to read (its
        // arrival must count for this filling of the slot, hence the wait).
        if (q < q1) {
          if (b == 0) {
            ok = wait_warp(B.lfull[s], ph_l);
            if (!ok) break;
            if (lane == 0) mbar_arrive(smem_u32(&B.lfree[s]));
          }
          continue;
        }
        const int n = ns++;
        if ((n & 1) != b) continue;
        ok = wait_warp(B.s[t][b], n / 2) && wait_warp(B.lfull[s], ph_l);
        if (!ok) break;
        tc_fence_after();
        const int toks = p.chunk - q * Jt;  // tokens from this tile on
        const bool all = q * Jt >= tmin_w && toks >= Jt;
        // Columns of tokens before tmin do not see the row; columns past the
        // chunk hold no query.
        const int c_lo = (tmin - q * Jt) * G, c_hi = min(Jt, toks) * G;
        uint64_t a0 = pk2(0.f, 0.f), a1 = a0;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          float e[2][32];
          tmem_ld32(tS + 64 * hf, e[0]);
          tmem_ld32(tS + 64 * hf + 32, e[1]);
          tmem_wait_ld();
          if (hf == 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&B.sfree[t][b]));
          }
          const ulonglong2 *nl = reinterpret_cast<const ulonglong2 *>(s_lse + s * kBlk + 64 * hf);
          if (all) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
              for (int x = 0; x < 32; x += 4) {
                const ulonglong2 z = nl[(32 * k + x) >> 2];
                float d0, d1, d2, d3;
                upk2(fma2(pk2(e[k][x], e[k][x + 1]), scale2, z.x), d0, d1);
                upk2(fma2(pk2(e[k][x + 2], e[k][x + 3]), scale2, z.y), d2, d3);
                a0 = add2(a0, pk2(ex2(d0), ex2(d1)));
                a1 = add2(a1, pk2(ex2(d2), ex2(d3)));
              }
          } else {
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
              for (int x = 0; x < 32; x += 4) {
                const ulonglong2 z = nl[(32 * k + x) >> 2];
                float d[4];
                upk2(fma2(pk2(e[k][x], e[k][x + 1]), scale2, z.x), d[0], d[1]);
                upk2(fma2(pk2(e[k][x + 2], e[k][x + 3]), scale2, z.y), d[2], d[3]);
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                  const int col = 64 * hf + 32 * k + x + y;
                  d[y] = col >= c_lo && col < c_hi ? ex2(d[y]) : 0.f;
                }
                a0 = add2(a0, pk2(d[0], d[1]));
                a1 = add2(a1, pk2(d[2], d[3]));
              }
          }
        }
        float x0, x1, y0, y1;
        upk2(a0, x0, x1);
        upk2(a1, y0, y1);
        sum += (x0 + x1) + (y0 + y1);
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&B.lfree[s]));
      }
      // The two warpgroups' sums, added one after the other.
      sum *= p.inv_g;
      float *su = c.score + it.u.ug * (size_t)c.sstride + slot;
      if (b == 0 && ok && slot < it.n) {
        const float before = *su;
        // For settling ties: behind the normalisers, which end before it.
        if (p.settle && slot < it.u.m)
          c.logits[(it.u.ug + 1) * (size_t)G * c.cap - it.u.m + slot] = before;
        *su = before + sum;
      }
      int bad;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
          "barrier.cta.red.or.pred q, %2, 256, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
          : "=r"(bad)
          : "r"(ok ? 0 : 1), "r"(1 + t)
          : "memory");
      if (bad) {
        ok = false;
        break;
      }
      if (b == 1 && slot < it.n) *su += sum;
    }
    if (!ok && lane == 0) {
      if (!*abort) atomicOr(c.err, ERR_TIMEOUT);
      *abort = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kProducer) tmem_dealloc(tm, kScCols);
}

}  // namespace

int absorb_long_box_rows() { return kBox; }

cudaError_t launch_absorb_long(const CUtensorMap &tmK, const CUtensorMap &tmV,
                               const CUtensorMap &tmQ, const AbsorbParams &p, int sms,
                               cudaStream_t st) {
  if (p.chunk < 1 || p.c.G > 8 || p.c.d != 128 || !p.c.kv_bf16 || !p.c.out_bf16)
    return cudaErrorInvalidValue;
  const int units = p.c.S * p.nl * p.c.H;
  const int Jt = kBlk / p.c.G, n_qt = (p.chunk + Jt - 1) / Jt;
  const int n_kp = (p.max_rows + 2 * kBlk - 1) / (2 * kBlk);
  cudaError_t e = cudaFuncSetAttribute(
      long_attend_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(long_score_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kScoreSmem);
  if (e != cudaSuccess) return e;
  // The logit scratch holds [u][G][cap] floats; a unit's normalisers take
  // chunk * G of its G * cap.
  float *lse = p.c.logits;
  e = launch_pdl(long_append_kernel,
                 dim3(units, min((p.chunk - 1) / kAppendRows + 1, kAppendCtas)), dim3(256), 0,
                 st, p);
  if (e != cudaSuccess) return e;
  const int n_att = units * n_qt, n_sc = units * n_kp;
  e = launch_pdl(long_attend_kernel, dim3(n_att < 2 * sms ? n_att : 2 * sms), dim3(kAttThr),
                 (size_t)kAttSmem, st, p, tmK, tmV, tmQ, lse, n_att, n_qt,
                 reinterpret_cast<uintptr_t>(p.out) % 32 == 0 ? 1 : 0);
  if (e != cudaSuccess) return e;
  return launch_pdl(long_score_kernel, dim3(n_sc < sms ? n_sc : sms), dim3(kScThr),
                    (size_t)kScoreSmem, st, p, tmK, tmQ, (const float *)lse, n_sc, n_qt);
}

}  // namespace kvr
