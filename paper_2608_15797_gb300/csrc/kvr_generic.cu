// kvr_generic.cu -- generic decode-step kernels of libkvr: one CTA per unit
// (sequence, layer, KV head), any head_dim in {64, 128}, G <= 8, fp32 or
// bf16 elements.  These serve every shape; the bf16 / d=128 steady state has
// a faster fused kernel (kvr_fused.cu).
//
// attend_score_kernel: Eq. 1 Attn(q_t, C) for the G query heads of one KV
//   head plus the accumulated-attention update of Sec. 2.1 (score += mean over
//   the G heads of the row's probability).  Logits live in shared memory when
//   they fit, else in the cache's per-unit logit scratch; K and V are each
//   read once.
// evict_kernel: TopB of Eq. 1 with the protected recent window of Sec. 4.1:
//   by rank where every row has a thread, else a histogram select of the B-th
//   best score among the non-window rows (ties to the lower position), then an
//   in-place compaction that moves the survivors lying beyond the new length
//   into the freed slots below it.  Long units are bound by the passes over
//   their rows: scores are kept in shared memory, the lists take two passes
//   and one exchange of counts (448 units of 700 to 16,384 rows: 152 us with
//   64-bit keys read from global memory eight times and block-wide list
//   building, 47 now; 1,792 units of 697 rows: 96 and 33, and 54 when a warp
//   moved one row at a time with half its lanes idle).
// tie_sums_kernel, evict_tied_kernel: the end of a blocked absorb
//   (kvr_absorb_long.cu) in units whose scores leave open which rows a
//   token-by-token absorb would keep.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "kvr_device.cuh"
#include "kvr_internal.h"

namespace kvr {
namespace {

using namespace dev;

struct Unit {
  int s, lr, l, h;
  size_t u;
};

__device__ __forceinline__ Unit unit_of(const CacheView &c, int lb, int nl) {
  Unit x;
  const int b = blockIdx.x;
  x.h = b % c.H;
  x.lr = (b / c.H) % nl;
  x.s = b / (c.H * nl);
  x.l = lb + x.lr;
  x.u = ((size_t)x.s * c.L + x.l) * c.H + x.h;
  return x;
}

// The need-th largest of v(i) over the rows i in [0, n) with v(i) != kNone, by
// passes over a 2,048-bin histogram, each over the range that the last one
// left: first the values' own range (scores share their leading bits, and
// bins by those would take all the additions), three passes at most.  Returns
// the value; *rest is how many of the rows that equal it belong to the `need`,
// *ties how many rows equal it.  need >= 1 and at least `need` such rows must
// exist.  lo, hi: the least and greatest value among the rows that this thread
// has seen (kNone, 0 for none); every row must have been seen by some thread.
// Every thread must call it.
constexpr unsigned kNone = 0xFFFFFFFFu;
struct SelectSmem {
  unsigned hist[2048];
  unsigned wsum[32], wmax[32];
  unsigned digit, above, count;
};
template <int NT, typename Val>
__device__ unsigned select_desc(int n, unsigned need, Val v, unsigned lo, unsigned hi,
                                SelectSmem &m, unsigned *rest, unsigned *ties) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kPer = 2048 / NT;  // bins a thread scans
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    m.wsum[warp] = lo;
    m.wmax[warp] = hi;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    lo = min(lo, m.wsum[w]);
    hi = max(hi, m.wmax[w]);
  }
  int shift = max(0, 32 - __clz((int)(hi - lo)) - 11);
  unsigned bins = 2048;  // of the range left
  for (bool last = false; !last;) {
    last = shift == 0;
    for (int i = tid; i < 2048; i += NT) m.hist[i] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += NT) {
      const unsigned x = v(i), bin = (x - lo) >> shift;
      if (x != kNone && bin < bins) atomicAdd(&m.hist[bin], 1u);
    }
    __syncthreads();
    // Inclusive counts from the top bin down; thread t owns kPer bins.
    unsigned c[kPer], s = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      c[k] = m.hist[2047 - (tid * kPer + k)];
      s += c[k];
    }
    unsigned inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) m.wsum[warp] = inc;
    __syncthreads();
    unsigned above = inc - s;
    for (int w = 0; w < warp; ++w) above += m.wsum[w];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      if (above < need && above + c[k] >= need) {
        m.digit = 2047 - (tid * kPer + k);
        m.above = above;
        m.count = c[k];
      }
      above += c[k];
    }
    __syncthreads();
    lo += m.digit << shift;
    need -= m.above;
    *ties = m.count;
    bins = 1u << min(shift, 11);
    shift = max(0, shift - 11);
    __syncthreads();
  }
  *rest = need;
  return lo;
}

// The end of an eviction: the rows that keep(i) names, nk of unit u's n, stay;
// lists has room for 2 * max_list entries.  Every thread must call it.
template <typename T, int D, int NT, typename Keep>
__device__ void compact_unit(const CacheView &c, size_t u, int n, int nk, Keep keep, int *lists,
                             int max_list, int2 *s_cnt) {
  const int tid = threadIdx.x;
  T *Ku = reinterpret_cast<T *>(c.K) + u * (size_t)c.cap * D;
  T *Vu = reinterpret_cast<T *>(c.V) + u * (size_t)c.cap * D;
  float *su = c.score + u * (size_t)c.sstride;
  int32_t *pu = c.pos + u * (size_t)c.sstride;
  int *holes = lists, *movers = lists + max_list;
  // The freed slots below nk and the survivors above, both in ascending
  // order: each warp takes a contiguous run of rows, counts, and after one
  // exchange of counts writes its part of the lists.
  constexpr int kNW = NT / 32;
  const int lane = tid & 31, warp = tid >> 5;
  const int seg = (n + kNW * 32 - 1) / (kNW * 32) * 32;
  const int r0 = min(n, warp * seg), r1 = min(n, r0 + seg);
  int ch = 0, cm = 0;
  for (int base = r0; base < r1; base += 32) {
    const int i = base + lane;
    const bool in = i < r1, k = in && keep(i);
    ch += __popc(__ballot_sync(0xffffffffu, in && i < nk && !k));
    cm += __popc(__ballot_sync(0xffffffffu, in && i >= nk && k));
  }
  if (lane == 0) s_cnt[warp] = make_int2(ch, cm);
  __syncthreads();
  int oh = 0, om = 0, nh = 0, nm = 0;
#pragma unroll
  for (int w = 0; w < kNW; ++w) {
    const int2 x = s_cnt[w];
    if (w < warp) {
      oh += x.x;
      om += x.y;
    }
    nh += x.x;
    nm += x.y;
  }
  // As many survivors above nk as free slots below: the window is intact
  // and B + W rows stay.
  if (nh != nm || nh > max_list) {
    if (tid == 0) atomicOr(c.err, ERR_LENGTH);
    return;
  }
  const unsigned below = (1u << lane) - 1u;
  for (int base = r0; base < r1; base += 32) {
    const int i = base + lane;
    const bool in = i < r1, k = in && keep(i);
    const bool h = in && i < nk && !k, m = in && i >= nk && k;
    const unsigned bh = __ballot_sync(0xffffffffu, h), bm = __ballot_sync(0xffffffffu, m);
    if (h) holes[oh + __popc(bh & below)] = i;
    if (m) movers[om + __popc(bm & below)] = i;
    oh += __popc(bh);
    om += __popc(bm);
  }
  __syncthreads();
  // Move every survivor beyond nk into a freed slot below it (disjoint), four
  // 16-byte pieces a thread in flight.
  for (int j = tid; j < nh; j += NT) {
    const int dst = holes[j], src = movers[j];
    su[dst] = su[src];
    pu[dst] = pu[src];
  }
  constexpr int kChunks = D * (int)sizeof(T) / 16, kAhead = 4;
  const int pieces = nh * 2 * kChunks;  // of a row's K, then of its V
  for (int i0 = tid; i0 < pieces; i0 += kAhead * NT) {
    int4 v[kAhead];
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      const int i = i0 + k * NT;
      if (i < pieces)
        v[k] = reinterpret_cast<const int4 *>(
            ((i / kChunks) & 1 ? Vu : Ku) + (size_t)movers[i / (2 * kChunks)] * D)[i % kChunks];
    }
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      const int i = i0 + k * NT;
      if (i < pieces)
        reinterpret_cast<int4 *>(((i / kChunks) & 1 ? Vu : Ku) +
                                 (size_t)holes[i / (2 * kChunks)] * D)[i % kChunks] = v[k];
    }
  }
  if (tid == 0) {
    c.state[4 * u] = nk;
    c.state[4 * u + 2] = 0;  // the R-KV key sum no longer matches
  }
}

// Dynamic shared memory of attend_score_kernel (floats).
__host__ __device__ constexpr int attend_fixed_floats(int D) {
  return kMaxG * D                           // q
         + (kThreads / (D / 2)) * kMaxG * D  // PV partials per row group
         + 2 * kMaxG;                        // max and 1/sum per head
}

// kExtScratch: logits always go to `ext`, one [G][max_rows] block per CTA,
// instead of shared memory or the cache's own scratch area.  kEvict: the CTA
// also cuts its unit (at most kThreads rows with the new one) back to budget +
// window rows, by rank, as evict_kernel would: one launch where a step's cost
// is launches (one layer, 2 units, fp32: 9.0 us a step in two, 6.9 in one).
template <typename T, typename O, int D, bool kExtScratch = false, bool kEvict = false>
__global__ void __launch_bounds__(kThreads)
    attend_score_kernel(CacheView c, StepArgs a, int logits_in_smem,
                        float *ext) {
  pdl_begin();
  extern __shared__ float smem[];
  constexpr int P = D / 2;         // dimension pairs
  constexpr int R = kThreads / P;  // row groups of the PV pass
  constexpr int E = D / 32;        // elements per lane in the QK pass
  float *qs = smem;
  float *red = qs + kMaxG * D;
  float *stat_m = red + R * kMaxG * D;
  float *stat_iz = stat_m + kMaxG;
  float *lg_s = stat_iz + kMaxG;

  const int G = c.G;
  const Unit x = unit_of(c, a.lb, a.nl);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  const int n0 = c.state[4 * x.u];
  if (n0 + 1 > c.cap) {
    if (tid == 0) atomicOr(c.err, ERR_CAPACITY);
    return;
  }
  const int n = n0 + 1;
  T *Ku = reinterpret_cast<T *>(c.K) + x.u * (size_t)c.cap * D;
  T *Vu = reinterpret_cast<T *>(c.V) + x.u * (size_t)c.cap * D;
  float *su = c.score + x.u * (size_t)c.sstride;
  int32_t *pu = c.pos + x.u * (size_t)c.sstride;
  const size_t kv_row =
      (((size_t)x.s * a.nl + x.lr) * a.chunk + a.tok) * c.H + x.h;
  const size_t q_row = kv_row * G;
  const T *qg = reinterpret_cast<const T *>(a.q) + q_row * D;
  const T *kn = reinterpret_cast<const T *>(a.k_new) + kv_row * D;
  const T *vn = reinterpret_cast<const T *>(a.v_new) + kv_row * D;

  // Append: the new row goes to slot n0 with score 0 and the next position.
  for (int i = tid; i < G * D; i += kThreads) qs[i] = to_f(qg[i]);
  for (int i = tid; i < D; i += kThreads) {
    Ku[(size_t)n0 * D + i] = kn[i];
    Vu[(size_t)n0 * D + i] = vn[i];
  }
  const int newest = c.state[4 * x.u + 1];
  if (tid == 0) {
    pu[n0] = newest;
    su[n0] = 0.f;
  }
  __syncthreads();

  float *lg = kExtScratch ? ext + (size_t)blockIdx.x * G * a.max_rows
              : logits_in_smem ? lg_s
                               : c.logits + x.u * (size_t)G * c.cap;
  const int ls = (kExtScratch || logits_in_smem) ? a.max_rows : c.cap;

  // Logits l_{g,i} = scale * <q_g, k_i>: one warp per row.
  for (int i = warp; i < n; i += kWarps) {
    const T *kr = Ku + (size_t)i * D + lane * E;
    float kv[E];
#pragma unroll
    for (int e = 0; e < E; e += 2) {
      float2 t = ld2(kr + e);
      kv[e] = t.x;
      kv[e + 1] = t.y;
    }
#pragma unroll
    for (int g = 0; g < kMaxG; ++g) {
      if (g < G) {
        const float acc = warp_sum(lane_dot<E>(qs + g * D + lane * E, kv));
        if (lane == 0) lg[(size_t)g * ls + i] = acc * c.scale;
      }
    }
  }
  __syncthreads();

  // Softmax statistics: warp g owns query head g.
  if (warp < G) {
    float m, z;
    warp_softmax(lg + (size_t)warp * ls, n, lane, m, z);
    if (lane == 0) {
      stat_m[warp] = m;
      stat_iz[warp] = 1.f / z;
      if (!(z >= 1.f) || !isfinite(z) || !isfinite(m)) atomicOr(c.err, ERR_NONFINITE);
    }
  }
  __syncthreads();

  // Probabilities, and the accumulated-attention update with their mean.
  const float inv_g = 1.f / (float)G;
  for (int i = tid; i < n; i += kThreads) {
    float acc = 0.f;
    for (int g = 0; g < G; ++g) {
      const float p = head_prob(lg[(size_t)g * ls + i], stat_m[g], stat_iz[g]);
      lg[(size_t)g * ls + i] = p;
      acc = __fadd_rn(acc, p);
    }
    su[i] = add_mean(su[i], acc, inv_g);
  }
  __syncthreads();

  // out_g = sum_i p_{g,i} v_i: thread (row group, dimension pair).
  const int dp = tid % P, rg = tid / P;
  float acc[kMaxG][2];
#pragma unroll
  for (int g = 0; g < kMaxG; ++g) acc[g][0] = acc[g][1] = 0.f;
  for (int i = rg; i < n; i += R) {
    const float2 v = ld2(Vu + (size_t)i * D + 2 * dp);
#pragma unroll
    for (int g = 0; g < kMaxG; ++g) {
      if (g < G) {
        const float p = lg[(size_t)g * ls + i];
        acc[g][0] += p * v.x;
        acc[g][1] += p * v.y;
      }
    }
  }
#pragma unroll
  for (int g = 0; g < kMaxG; ++g) {
    red[(rg * kMaxG + g) * D + 2 * dp] = acc[g][0];
    red[(rg * kMaxG + g) * D + 2 * dp + 1] = acc[g][1];
  }
  __syncthreads();
  O *og = reinterpret_cast<O *>(a.out) + q_row * D;
  for (int i = tid; i < G * D; i += kThreads) {
    const int g = i / D, dd = i % D;
    float o = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) o += red[(r * kMaxG + g) * D + dd];
    st1(og + i, o);
  }
  if (tid == 0) {
    c.state[4 * x.u] = n;
    c.state[4 * x.u + 1] = newest + 1;
    c.state[4 * x.u + 2] = 0;  // the R-KV key sum no longer matches
  }
  if constexpr (kEvict) {
    const int nk = a.budget + a.window;
    if (n <= nk) return;
    if (n > kThreads) {  // the host sized the launch from its mirror
      if (tid == 0) atomicOr(c.err, ERR_LENGTH);
      return;
    }
    __shared__ unsigned long long s_key[kThreads];
    __shared__ unsigned char s_keep[kThreads];
    __shared__ int s_lists[2 * kThreads];
    __shared__ int2 s_cnt[kWarps];
    const int wlo = newest - a.window;
    block_rank_keep(
        n, a.budget, [&](int i) { return pu[i] <= wlo; },
        [&](int i) { return rank_key(su[i], pu[i]); }, s_key, s_keep);
    compact_unit<T, D, kThreads>(
        c, x.u, n, nk, [&](int i) { return s_keep[i] != 0; }, s_lists, kThreads, s_cnt);
  }
}

// A near tie: the least score kept and the greatest dropped lie closer than the
// blocked absorb's sums are certain to, so which of the rows around the cut a
// token-by-token absorb would keep is not known.  Lists those rows and enters
// the unit in the call's list; false where there is no tie, or one of more than
// kMaxTied rows (whose scores are as a rule equal to the bit on either path).
// val(i): a candidate's score bits, kNone for the window's rows; keep(i): as the
// scores stand.  Every thread must call it.
template <int NT, typename Val, typename Keep>
__device__ bool near_tie(const CacheView &c, int lb, int nl, size_t u, int n, int chunk,
                         float band, Val val, Keep keep) {
  __shared__ unsigned s_lo[NT / 32], s_hi[NT / 32];
  __shared__ int s_n;
  const int tid = threadIdx.x;
  unsigned lo = kNone, hi = 0;
  for (int i = tid; i < n; i += NT) {
    const unsigned b = val(i);
    if (b == kNone) continue;
    if (keep(i)) lo = min(lo, b);
    else hi = max(hi, b);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((tid & 31) == 0) {
    s_lo[tid >> 5] = lo;
    s_hi[tid >> 5] = hi;
  }
  if (tid == 0) s_n = 0;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    lo = min(lo, s_lo[w]);
    hi = max(hi, s_hi[w]);
  }
  const float least = __uint_as_float(lo), most = __uint_as_float(hi), w = band * least;
  if (lo == kNone || !(least - most <= w)) return false;
  int *words = tie_words(c, u);
  for (int i = tid; i < n; i += NT) {
    const unsigned b = val(i);
    const float x = __uint_as_float(b);
    if (b != kNone && x >= most - w && x <= least + w) {
      const int k = atomicAdd(&s_n, 1);
      if (k < kMaxTied) words[kTieRows + k] = i;
    }
  }
  __syncthreads();
  const int nt = s_n;
  if (nt > kMaxTied) return false;
  if (tid == 0) {
    words[kTieCount] = nt;
    const int e = atomicAdd(&tie_words(c, unit_index(c, lb, nl, 0))[kTieUnits], 1);
    tie_words(c, unit_index(c, lb, nl, e))[kTieEntry] = blockIdx.x;
  }
  return true;
}

// Cut a unit of n > B + W rows back to B + W.  kByRank: units of at most NT
// rows, one row a thread, kept by rank; otherwise the B-th best score is
// selected over the unit's scores, which shared memory holds once (`cached`;
// else they are read from global memory on every pass).  tied(val, keep) is
// asked first, and true leaves the unit as it is.  Every thread must call it.
template <typename T, int D, int NT, bool kByRank, typename Tied>
__device__ void evict_unit(const CacheView &c, size_t u, int n, int newest, int B, int W,
                           int *lists, int max_list, int cached, Tied tied) {
  __shared__ unsigned s_wsum[NT / 32];
  __shared__ int2 s_cnt[NT / 32];
  const int tid = threadIdx.x;
  float *su = c.score + u * (size_t)c.sstride;
  int32_t *pu = c.pos + u * (size_t)c.sstride;
  // The W most recent positions are protected; a row is a candidate iff its
  // position is at most newest - W.
  const int wlo = newest - W;
  // A candidate's score bits (scores are >= 0: they order like the values),
  // kNone for the window's rows.
  auto bits = [&](int i) {
    return pu[i] <= wlo ? min(__float_as_uint(su[i]), kNone - 1) : kNone;
  };
  auto finish = [&](auto val, auto keep) {
    if (tied(val, keep)) return;
    compact_unit<T, D, NT>(c, u, n, B + W, keep, lists, max_list, s_cnt);
  };
  if constexpr (kByRank) {
    __shared__ unsigned long long s_key[NT];
    __shared__ unsigned char s_keep[NT];
    block_rank_keep(
        n, B, [&](int i) { return pu[i] <= wlo; },
        [&](int i) { return rank_key(su[i], pu[i]); }, s_key, s_keep);
    finish(bits, [&](int i) { return s_keep[i] != 0; });
  } else {
    __shared__ SelectSmem m;
    unsigned *sv = reinterpret_cast<unsigned *>(lists + 2 * max_list);
    int have = 0;
    unsigned lo = kNone, hi = 0;
    for (int i0 = tid; i0 < n; i0 += 4 * NT) {  // four rows' loads in flight
      int32_t ps[4];
      float sc[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = i0 + k * NT;
        ps[k] = i < n ? pu[i] : INT32_MAX;
        sc[k] = i < n ? su[i] : 0.f;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = i0 + k * NT;
        const bool cand = i < n && ps[k] <= wlo;
        const unsigned b = cand ? min(__float_as_uint(sc[k]), kNone - 1) : kNone;
        if (cached && i < n) sv[i] = b;
        lo = min(lo, b);
        if (cand) hi = max(hi, b);
        have += cand ? 1 : 0;
      }
    }
    have = __reduce_add_sync(0xffffffffu, have);
    if ((tid & 31) == 0) s_wsum[tid >> 5] = have;
    __syncthreads();
    have = 0;
    for (int w = 0; w < NT / 32; ++w) have += (int)s_wsum[w];
    __syncthreads();
    auto val = [&](int i) { return cached ? sv[i] : bits(i); };
    unsigned thr = 0, last = 0;  // scores above thr stay; ties at positions up to ~last
    if (B > 0 && have > B) {
      unsigned rest, ties;
      thr = select_desc<NT>(n, (unsigned)B, val, lo, hi, m, &rest, &ties);
      if (rest < ties) {
        // Equal scores: the lower positions stay.
        unsigned r2, t2;
        auto low_pos = [&](int i) { return val(i) == thr ? ~(unsigned)pu[i] - 1u : kNone; };
        lo = kNone;
        hi = 0;
        for (int i = tid; i < n; i += NT) {
          const unsigned b = low_pos(i);
          lo = min(lo, b);
          if (b != kNone) hi = max(hi, b);
        }
        last = select_desc<NT>(n, rest, low_pos, lo, hi, m, &r2, &t2);
      }
    }
    finish(val, [&](int i) {
      const unsigned b = val(i);
      if (b == kNone) return true;
      if (B == 0) return false;
      return b > thr || (b == thr && ~(unsigned)pu[i] - 1u >= last);
    });
  }
}

// Cut every unit longer than B + W back to B + W rows.  kTies (the blocked
// absorb of `grow` tokens): units with a near tie are listed and left long.
template <typename T, int D, int NT, bool kByRank, bool kTies>
__global__ void __launch_bounds__(NT)
    evict_kernel(CacheView c, int lb, int nl, int B, int W, int grow, int max_list,
                 int cached, int max_rows, float band) {
  pdl_begin();
  extern __shared__ int lists[];  // holes | movers [max_list each] | scores

  const Unit x = unit_of(c, lb, nl);
  const int tid = threadIdx.x;
  // `grow` rows were appended whose length is not recorded yet.
  const int n = c.state[4 * x.u] + grow;
  const int newest = c.state[4 * x.u + 1] + grow - 1;
  __syncthreads();
  // Longer than the host thinks: the blocked absorb left such a unit alone, and
  // an eviction has no room for its lists.
  if (n < grow || n > (grow ? min(max_rows, c.cap) : max(max_rows, B + W))) {
    if (tid == 0) atomicOr(c.err, ERR_LENGTH);
    return;
  }
  if (tid == 0 && grow) {
    c.state[4 * x.u] = n;
    c.state[4 * x.u + 1] = newest + 1;
    c.state[4 * x.u + 2] = 0;  // the R-KV key sum no longer matches
  }
  if (n <= B + W) return;
  evict_unit<T, D, NT, kByRank>(c, x.u, n, newest, B, W, lists, max_list, cached,
                                [&](auto val, auto keep) {
                                  if constexpr (kTies)
                                    return near_tie<NT>(c, lb, nl, x.u, n, grow, band, val, keep);
                                  return false;
                                });
}

// Of token `tok` of a blocked absorb: put(i, x) with x the sum over the heads of
// the probabilities of the unit's i-th tied row, by the arithmetic of
// attend_score_kernel to the bit: a warp a row, its lanes' products summed over
// the same offsets (the heads' sums are folded into each other, so that the five
// steps take 9 exchanges for eight heads).  smem: tie_smem() bytes.  Every
// thread must call it.
template <typename Put>
__device__ void tie_sums(const AbsorbParams &p, int x, int tok, float *smem, Put put) {
  __shared__ float s_m[kMaxG], s_iz[kMaxG];
  const CacheView &c = p.c;
  const int G = c.G, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x;
  float *lg = smem;  // [G][max_rows]
  const size_t u = unit_index(c, p.lb, p.nl, x);
  const int n = c.state[4 * u] - p.chunk + tok + 1;  // rows that the token sees
  auto row4 = [](uint2 w, float(&v)[4]) {
    v[0] = __uint_as_float(w.x << 16);
    v[1] = __uint_as_float(w.x & 0xFFFF0000u);
    v[2] = __uint_as_float(w.y << 16);
    v[3] = __uint_as_float(w.y & 0xFFFF0000u);
  };
  const uint2 *Q = reinterpret_cast<const uint2 *>(p.q) +
                   (((size_t)(x / c.H) * p.chunk + tok) * c.H + x % c.H) * (size_t)G * 32;
  const uint2 *K = reinterpret_cast<const uint2 *>(c.K) + u * (size_t)c.cap * 32;
  float q[kMaxG][4];
#pragma unroll
  for (int h = 0; h < kMaxG; ++h) row4(h < G ? Q[h * 32 + lane] : make_uint2(0u, 0u), q[h]);
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  const int g = lane >> 2;  // the head whose sum this lane ends with
  constexpr int kAhead = 8;  // rows a warp has in flight
  for (int i0 = warp; i0 < n; i0 += kAhead * (NT / 32)) {
    uint2 kw[kAhead];
#pragma unroll
    for (int r = 0; r < kAhead; ++r) {
      const int i = i0 + r * (NT / 32);
      kw[r] = i < n ? K[(size_t)i * 32 + lane] : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int r = 0; r < kAhead; ++r) {
      const int i = i0 + r * (NT / 32);
      float k[4], a[kMaxG];
      row4(kw[r], k);
#pragma unroll
      for (int h = 0; h < kMaxG; ++h) a[h] = lane_dot<4>(q[h], k);
#pragma unroll
      for (int h = 0; h < 4; ++h)
        a[h] = (b4 ? a[h + 4] : a[h]) + __shfl_xor_sync(0xffffffffu, b4 ? a[h] : a[h + 4], 16);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        a[h] = (b3 ? a[h + 2] : a[h]) + __shfl_xor_sync(0xffffffffu, b3 ? a[h] : a[h + 2], 8);
      float s = (b2 ? a[1] : a[0]) + __shfl_xor_sync(0xffffffffu, b2 ? a[0] : a[1], 4);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      if (i < n && (lane & 3) == 0 && g < G) lg[(size_t)g * p.max_rows + i] = s * c.scale;
    }
  }
  __syncthreads();
  if (warp < G) {
    float m, z;
    warp_softmax(lg + (size_t)warp * p.max_rows, n, lane, m, z);
    if (lane == 0) {
      s_m[warp] = m;
      s_iz[warp] = 1.f / z;
    }
  }
  __syncthreads();
  const int *words = tie_words(c, u);
  for (int i = tid; i < words[kTieCount]; i += NT) {
    const int slot = words[kTieRows + i];
    float sum = 0.f;
    if (slot < n)
      for (int h = 0; h < G; ++h)
        sum = __fadd_rn(sum, head_prob(lg[(size_t)h * p.max_rows + slot], s_m[h], s_iz[h]));
    put(i, sum);
  }
  __syncthreads();
}
size_t tie_smem(const CacheView &c, int max_rows) {
  return (size_t)c.G * max_rows * sizeof(float);
}

// Those sums for every listed unit, one CTA a token and unit.  Few units have
// ties, and a launch that finds none ends at once.
__global__ void __launch_bounds__(kThreads) tie_sums_kernel(const AbsorbParams p) {
  pdl_begin();
  extern __shared__ __align__(16) float tie_mem[];
  const CacheView &c = p.c;
  const int count = tie_words(c, unit_index(c, p.lb, p.nl, 0))[kTieUnits];
  for (long long job = blockIdx.x; job < (long long)count * p.chunk; job += gridDim.x) {
    const int e = (int)(job / p.chunk), tok = (int)(job % p.chunk);
    const int x = tie_words(c, unit_index(c, p.lb, p.nl, e))[kTieEntry];
    const size_t u = unit_index(c, p.lb, p.nl, x);
    if (!tie_room(c, tie_words(c, u)[kTieCount], p.chunk, c.state[4 * u] - p.chunk)) continue;
    float *sums = c.logits + u * (size_t)c.G * c.cap;
    const int tied = tie_words(c, u)[kTieCount];
    tie_sums(p, x, tok, tie_mem, [&](int i, float sum) { sums[(size_t)tok * tied + i] = sum; });
  }
}

// The listed units, one a CTA at a time: the tied rows' scores, token by token
// as attend_score_kernel adds them (the sums formed here where the unit's
// scratch, at G = 1 or 2, had no room for them), then the eviction.
template <typename T, int D, int NT, bool kByRank>
__global__ void __launch_bounds__(NT)
    evict_tied_kernel(const AbsorbParams p, int B, int W, int max_list, int cached) {
  pdl_begin();
  extern __shared__ __align__(16) float tie_mem[];  // tie_sums' or evict_unit's
  int *lists = reinterpret_cast<int *>(tie_mem);
  __shared__ float s_score[kMaxTied];
  const CacheView &c = p.c;
  const int count = tie_words(c, unit_index(c, p.lb, p.nl, 0))[kTieUnits];
  for (int e = blockIdx.x; e < count; e += gridDim.x) {
    const int x = tie_words(c, unit_index(c, p.lb, p.nl, e))[kTieEntry];
    const size_t u = unit_index(c, p.lb, p.nl, x);
    const int *words = tie_words(c, u);
    const int n = c.state[4 * u], newest = c.state[4 * u + 1] - 1, m = n - p.chunk;
    const int tied = words[kTieCount];
    const float *sums = c.logits + u * (size_t)c.G * c.cap;
    const float *old = sums + (size_t)c.G * c.cap - m;
    const bool room = tie_room(c, tied, p.chunk, m);
    for (int i = threadIdx.x; i < tied; i += NT) {
      const int slot = words[kTieRows + i];
      float s = slot < m ? old[slot] : 0.f;
      if (room) {
#pragma unroll 32
        for (int j = 0; j < p.chunk; ++j)  // (0 from a token that does not see the row)
          s = add_mean(s, sums[(size_t)j * tied + i], p.inv_g);
      }
      s_score[i] = s;
    }
    if (!room)
      for (int j = 0; j < p.chunk; ++j)
        tie_sums(p, x, j, tie_mem, [&](int i, float sum) {
          s_score[i] = add_mean(s_score[i], sum, p.inv_g);
        });
    for (int i = threadIdx.x; i < tied; i += NT)  // (each thread its own)
      c.score[u * (size_t)c.sstride + words[kTieRows + i]] = s_score[i];
    __syncthreads();
    evict_unit<T, D, NT, kByRank>(c, u, n, newest, B, W, lists, max_list, cached,
                                  [](auto, auto) { return false; });
    __syncthreads();
  }
}

// Copy one sequence's prompt rows [L][H][n][d] into its slabs.
template <typename T, int D>
__global__ void load_kernel(CacheView c, int seq, const T *k, const T *v,
                            int n, int first_pos) {
  const int lh = blockIdx.x;  // layer * H + head
  const size_t u = (size_t)seq * c.L * c.H + lh;
  const int r0 = blockIdx.y * 32;
  const int r1 = min(r0 + 32, n);
  T *Ku = reinterpret_cast<T *>(c.K) + u * (size_t)c.cap * D;
  T *Vu = reinterpret_cast<T *>(c.V) + u * (size_t)c.cap * D;
  const T *ks = k + (size_t)lh * n * D;
  const T *vs = v + (size_t)lh * n * D;
  constexpr int kChunks = D * (int)sizeof(T) / 16;
  for (int q = threadIdx.x; q < (r1 - r0) * kChunks; q += blockDim.x) {
    const size_t r = r0 + q / kChunks, cidx = q % kChunks;
    reinterpret_cast<int4 *>(Ku + r * D)[cidx] =
        reinterpret_cast<const int4 *>(ks + r * D)[cidx];
    reinterpret_cast<int4 *>(Vu + r * D)[cidx] =
        reinterpret_cast<const int4 *>(vs + r * D)[cidx];
  }
  for (int r = r0 + threadIdx.x; r < r1; r += blockDim.x) {
    c.score[u * c.sstride + r] = 0.f;
    c.pos[u * c.sstride + r] = first_pos + r;
  }
  if (blockIdx.y == 0 && threadIdx.x == 0) {
    c.state[4 * u] = n;
    c.state[4 * u + 1] = first_pos + n;
    c.state[4 * u + 2] = 0;  // no R-KV key sum yet
  }
}

template <typename T, typename O, int D>
cudaError_t attend_dispatch(const CacheView &c, const StepArgs &a,
                            cudaStream_t st) {
  const size_t fixed = attend_fixed_floats(D) * sizeof(float);
  const size_t lg = (size_t)kMaxG * a.max_rows * sizeof(float);
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const int in_smem = fixed + lg <= (size_t)optin ? 1 : 0;
  const size_t bytes = fixed + (in_smem ? lg : 0);
  auto kern = a.evict ? attend_score_kernel<T, O, D, false, true>
                      : attend_score_kernel<T, O, D>;
  cudaError_t e = cudaFuncSetAttribute(
      kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  const int grid = c.S * a.nl * c.H;
  return launch_pdl(kern, dim3(grid), dim3(kThreads), bytes, st, c, a, in_smem,
                    static_cast<float *>(nullptr));
}

template <typename T, typename O, int D>
cudaError_t attend_ext_dispatch(const CacheView &c, const StepArgs &a,
                                float *ext, cudaStream_t st) {
  const size_t bytes = attend_fixed_floats(D) * sizeof(float);
  auto kern = attend_score_kernel<T, O, D, true>;
  cudaError_t e = cudaFuncSetAttribute(
      kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(c.S * a.nl * c.H), dim3(kThreads), bytes, st, c,
                    a, 0, ext);
}

// Rows a CTA of the radix select keeps in shared memory, and the rows from
// which a unit takes 1,024 threads instead of 256 (few units, long scans).
constexpr int kCachedRows = 49152, kWideRows = 2048;

// An eviction's launch: the kernel's threads a unit and whether it ranks, by the
// longest unit, and its shared memory.
template <typename Run>
cudaError_t evict_shape(int max_rows, int nk, Run run) {
  const int max_list = std::max(1, std::min(nk, max_rows - nk));
  const bool by_rank = max_rows <= kThreads;
  const int cached = !by_rank && max_rows <= kCachedRows &&
                     (2 * (size_t)max_list + max_rows) * sizeof(int) <= 200 * 1024;
  const size_t bytes = (2 * (size_t)max_list + (cached ? max_rows : 0)) * sizeof(int);
  using std::integral_constant;
  if (by_rank)
    return run(integral_constant<int, kThreads>{}, std::true_type{}, max_list, cached, bytes);
  if (max_rows <= kWideRows)
    return run(integral_constant<int, kThreads>{}, std::false_type{}, max_list, cached, bytes);
  return run(integral_constant<int, 1024>{}, std::false_type{}, max_list, cached, bytes);
}

template <typename T, int D, bool kTies = false>
cudaError_t evict_dispatch(const CacheView &c, int lb, int nl, int max_rows, int B, int W,
                           int grow, cudaStream_t st, float band = 0.f) {
  return evict_shape(max_rows, B + W, [&](auto nt, auto rank, int max_list, int cached,
                                          size_t bytes) {
    constexpr int NT = decltype(nt)::value;
    auto kern = evict_kernel<T, D, NT, decltype(rank)::value, kTies>;
    const cudaError_t e = cudaFuncSetAttribute(
        kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, dim3(c.S * nl * c.H), dim3(NT), bytes, st, c, lb, nl, B, W, grow,
                      max_list, cached, max_rows, band);
  });
}

}  // namespace

int generic_evict_rows() { return kThreads; }

cudaError_t launch_attend_score_generic(const CacheView &c, const StepArgs &a,
                                        cudaStream_t st) {
  if (c.kv_bf16) {
    if (c.d == 128)
      return c.out_bf16
                 ? attend_dispatch<__nv_bfloat16, __nv_bfloat16, 128>(c, a, st)
                 : attend_dispatch<__nv_bfloat16, float, 128>(c, a, st);
    return c.out_bf16
               ? attend_dispatch<__nv_bfloat16, __nv_bfloat16, 64>(c, a, st)
               : attend_dispatch<__nv_bfloat16, float, 64>(c, a, st);
  }
  if (c.d == 128)
    return c.out_bf16 ? attend_dispatch<float, __nv_bfloat16, 128>(c, a, st)
                      : attend_dispatch<float, float, 128>(c, a, st);
  return c.out_bf16 ? attend_dispatch<float, __nv_bfloat16, 64>(c, a, st)
                    : attend_dispatch<float, float, 64>(c, a, st);
}

cudaError_t launch_attend_score_ext_scratch(const CacheView &c,
                                            const StepArgs &a, float *ext,
                                            cudaStream_t st) {
  if (c.kv_bf16) {
    if (c.d == 128)
      return c.out_bf16 ? attend_ext_dispatch<__nv_bfloat16, __nv_bfloat16,
                                              128>(c, a, ext, st)
                        : attend_ext_dispatch<__nv_bfloat16, float, 128>(
                              c, a, ext, st);
    return c.out_bf16
               ? attend_ext_dispatch<__nv_bfloat16, __nv_bfloat16, 64>(c, a,
                                                                        ext, st)
               : attend_ext_dispatch<__nv_bfloat16, float, 64>(c, a, ext, st);
  }
  if (c.d == 128)
    return c.out_bf16
               ? attend_ext_dispatch<float, __nv_bfloat16, 128>(c, a, ext, st)
               : attend_ext_dispatch<float, float, 128>(c, a, ext, st);
  return c.out_bf16 ? attend_ext_dispatch<float, __nv_bfloat16, 64>(c, a, ext, st)
                    : attend_ext_dispatch<float, float, 64>(c, a, ext, st);
}

cudaError_t launch_evict_generic(const CacheView &c, int lb, int nl,
                                 int max_rows, int budget, int window,
                                 cudaStream_t st, int grow) {
  if (c.kv_bf16)
    return c.d == 128
               ? evict_dispatch<__nv_bfloat16, 128>(c, lb, nl, max_rows, budget,
                                                    window, grow, st)
               : evict_dispatch<__nv_bfloat16, 64>(c, lb, nl, max_rows, budget,
                                                   window, grow, st);
  return c.d == 128 ? evict_dispatch<float, 128>(c, lb, nl, max_rows, budget,
                                                 window, grow, st)
                    : evict_dispatch<float, 64>(c, lb, nl, max_rows, budget,
                                                window, grow, st);
}

// Scores of the blocked absorb and of the token-by-token one differ by the order
// of their sums, one rounding a token on the latter's side: near the cut by
// 1.3e-7 rms and 7.3e-7 at most after 57 tokens (7B, 16 sequences of 640 rows,
// three inputs; 4.6e-7 after 10), 5.7e-7 and 2.5e-6 after 1,000.  Two rows'
// order is taken as certain beyond 1.2e-6, six times the rms of two rows'
// difference (and five times after 1,000 tokens: 4.7e-6).  Settling one to four
// tied units is 28 us for the sums and 13 for the rest of 768; without ties the
// launches are 12 of 741, and a prompt of 1,000 tokens with a tied unit takes
// 0.1 ms more than 0.92.
float tie_band(int chunk) { return 0x1.4p-20f * std::max(1.f, std::sqrt(chunk / 64.f)); }

bool can_settle(const CacheView &c, int max_rows) {
  return tie_smem(c, max_rows) <= 200 * 1024;
}

cudaError_t launch_evict_absorbed(const AbsorbParams &p, int budget, int window, int sms,
                                  cudaStream_t st) {
  using T = __nv_bfloat16;
  const CacheView &c = p.c;
  cudaError_t e = evict_dispatch<T, 128, true>(c, p.lb, p.nl, p.max_rows, budget, window,
                                               p.chunk, st, tie_band(p.chunk));
  if (e != cudaSuccess) return e;
  const size_t sums = tie_smem(c, p.max_rows);
  e = cudaFuncSetAttribute(tie_sums_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)sums);
  if (e == cudaSuccess)
    e = launch_pdl(tie_sums_kernel, dim3(4 * sms), dim3(kThreads), sums, st, p);
  if (e != cudaSuccess) return e;
  return evict_shape(p.max_rows, budget + window, [&](auto nt, auto rank, int max_list,
                                                      int cached, size_t lists) {
    constexpr int NT = decltype(nt)::value;
    auto kern = evict_tied_kernel<T, 128, NT, decltype(rank)::value>;
    const size_t bytes = std::max(lists, sums);
    const cudaError_t e1 = cudaFuncSetAttribute(
        kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e1 != cudaSuccess) return e1;
    return launch_pdl(kern, dim3(std::min(c.S * p.nl * c.H, sms)), dim3(NT), bytes, st, p,
                      budget, window, max_list, cached);
  });
}

cudaError_t launch_load(const CacheView &c, int seq, const void *k,
                        const void *v, int n_rows, int first_pos,
                        cudaStream_t st) {
  // At least one row-block so that an empty prompt still resets the length.
  dim3 grid(c.L * c.H, n_rows > 0 ? (n_rows + 31) / 32 : 1);
  if (c.kv_bf16) {
    if (c.d == 128)
      load_kernel<__nv_bfloat16, 128><<<grid, 256, 0, st>>>(
          c, seq, (const __nv_bfloat16 *)k, (const __nv_bfloat16 *)v, n_rows,
          first_pos);
    else
      load_kernel<__nv_bfloat16, 64><<<grid, 256, 0, st>>>(
          c, seq, (const __nv_bfloat16 *)k, (const __nv_bfloat16 *)v, n_rows,
          first_pos);
  } else {
    if (c.d == 128)
      load_kernel<float, 128><<<grid, 256, 0, st>>>(
          c, seq, (const float *)k, (const float *)v, n_rows, first_pos);
    else
      load_kernel<float, 64><<<grid, 256, 0, st>>>(
          c, seq, (const float *)k, (const float *)v, n_rows, first_pos);
  }
  return cudaGetLastError();
}

cudaError_t launch_init(const CacheView &c, cudaStream_t st) {
  const size_t units = (size_t)c.S * c.L * c.H;
  cudaError_t e = cudaMemsetAsync(c.state, 0, units * 4 * sizeof(int32_t), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(c.err, 0, 16, st);
  return e;
}

}  // namespace kvr
