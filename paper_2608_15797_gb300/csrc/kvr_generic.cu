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
#include <cuda_bf16.h>
#include <math.h>

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
        float acc = 0.f;
#pragma unroll
        for (int e = 0; e < E; ++e) acc += qs[g * D + lane * E + e] * kv[e];
        acc = warp_sum(acc);
        if (lane == 0) lg[(size_t)g * ls + i] = acc * c.scale;
      }
    }
  }
  __syncthreads();

  // Softmax statistics: warp g owns query head g.
  if (warp < G) {
    const float *lr = lg + (size_t)warp * ls;
    float m = -INFINITY;
    for (int i = lane; i < n; i += 32) m = fmaxf(m, lr[i]);
    m = warp_max(m);
    float z = 0.f;
    for (int i = lane; i < n; i += 32) z += expf(lr[i] - m);
    z = warp_sum(z);
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
      const float p = expf(lg[(size_t)g * ls + i] - stat_m[g]) * stat_iz[g];
      lg[(size_t)g * ls + i] = p;
      acc += p;
    }
    su[i] += acc * inv_g;
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

// Cut every unit longer than B + W back to B + W rows.  kByRank: units of at
// most NT rows, one row a thread, kept by rank; otherwise the B-th best score
// is selected over the unit's scores, which shared memory holds once
// (`cached`; else they are read from global memory on every pass).
template <typename T, int D, int NT, bool kByRank>
__global__ void __launch_bounds__(NT)
    evict_kernel(CacheView c, int lb, int nl, int B, int W, int grow, int max_list,
                 int cached, int max_rows) {
  pdl_begin();
  extern __shared__ int lists[];  // holes | movers [max_list each] | scores
  __shared__ unsigned s_wsum[NT / 32];
  __shared__ int2 s_cnt[NT / 32];

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
  float *su = c.score + x.u * (size_t)c.sstride;
  int32_t *pu = c.pos + x.u * (size_t)c.sstride;
  // The W most recent positions are protected; a row is a candidate iff its
  // position is at most newest - W.
  const int wlo = newest - W;
  auto finish = [&](auto keep) {
    compact_unit<T, D, NT>(c, x.u, n, B + W, keep, lists, max_list, s_cnt);
  };
  if constexpr (kByRank) {
    __shared__ unsigned long long s_key[NT];
    __shared__ unsigned char s_keep[NT];
    block_rank_keep(
        n, B, [&](int i) { return pu[i] <= wlo; },
        [&](int i) { return rank_key(su[i], pu[i]); }, s_key, s_keep);
    finish([&](int i) { return s_keep[i] != 0; });
  } else {
    __shared__ SelectSmem m;
    unsigned *sv = reinterpret_cast<unsigned *>(lists + 2 * max_list);
    // A candidate's score bits (scores are >= 0: they order like the values),
    // kNone for the window's rows.
    auto bits = [&](int i) {
      return pu[i] <= wlo ? min(__float_as_uint(su[i]), kNone - 1) : kNone;
    };
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
    finish([&](int i) {
      const unsigned b = val(i);
      if (b == kNone) return true;
      if (B == 0) return false;
      return b > thr || (b == thr && ~(unsigned)pu[i] - 1u >= last);
    });
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

template <typename T, int D, int NT, bool kByRank>
cudaError_t evict_launch(const CacheView &c, int lb, int nl, int max_rows, int B, int W,
                         int grow, cudaStream_t st) {
  const int nk = B + W;
  const int max_list = max(1, min(nk, max_rows - nk));
  const int cached = !kByRank && max_rows <= kCachedRows &&
                     (2 * (size_t)max_list + max_rows) * sizeof(int) <= 200 * 1024;
  const size_t bytes = (2 * (size_t)max_list + (cached ? max_rows : 0)) * sizeof(int);
  auto kern = evict_kernel<T, D, NT, kByRank>;
  cudaError_t e = cudaFuncSetAttribute(
      kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(c.S * nl * c.H), dim3(NT), bytes, st, c, lb, nl, B, W, grow,
                    max_list, cached, max_rows);
}

template <typename T, int D>
cudaError_t evict_dispatch(const CacheView &c, int lb, int nl, int max_rows,
                           int B, int W, int grow, cudaStream_t st) {
  if (max_rows <= kThreads)
    return evict_launch<T, D, kThreads, true>(c, lb, nl, max_rows, B, W, grow, st);
  if (max_rows <= kWideRows)
    return evict_launch<T, D, kThreads, false>(c, lb, nl, max_rows, B, W, grow, st);
  return evict_launch<T, D, 1024, false>(c, lb, nl, max_rows, B, W, grow, st);
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
