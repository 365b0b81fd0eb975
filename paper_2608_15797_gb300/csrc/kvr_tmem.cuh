// kvr_tmem.cuh -- helpers of the kernels that keep logits, probabilities and
// outputs in tensor memory: wide TMEM loads and stores, MMAs with their A
// operand in TMEM, and a query row's attention on its own.
#pragma once

#include "kvr_ptx.cuh"

namespace kvr {
namespace ptx {

// 32 consecutive TMEM columns of this thread's lane (no wait).
__device__ __forceinline__ void tmem_ld32(uint32_t ta, float (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,"
      "%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, "
      "[%32];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]),
        "=f"(v[6]), "=f"(v[7]), "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]),
        "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]), "=f"(v[16]), "=f"(v[17]),
        "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]),
        "=f"(v[24]), "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]),
        "=f"(v[30]), "=f"(v[31])
      : "r"(ta));
}
__device__ __forceinline__ void tmem_st32(uint32_t ta, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,"
      "%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,"
      "%32};" ::"r"(ta),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]),
      "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]),
      "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]),
      "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
      "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t ta, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,"
      "%12,%13,%14,%15,%16};" ::"r"(ta),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]),
      "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]),
      "r"(v[14]), "r"(v[15])
      : "memory");
}
// 32 bytes to global memory, one whole sector a thread (32-byte aligned).
__device__ __forceinline__ void st_global32(void *dst, const uint32_t *v) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dst), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// D[tmem] (+)= A[tmem] * B[smem], issued by one thread.
__device__ __forceinline__ void tc_mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t id,
                                          bool acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
      "r"(a), "l"(b), "r"(id), "r"(acc ? 1 : 0)
      : "memory");
}

// One query row on its own, over the n rows it sees of K and V (128 bf16 a row):
// o[x] += 2^(q.k scale - ref) v[c0 + x].  For the rows of a tile whose outputs are
// not finite: the rows that a tile's mask hides have P = 0 in its product with
// V, and 0 x NaN or 0 x Inf there is NaN, so a row that another query (a
// later token's, another candidate's) put a non-finite value in would reach
// queries that do not see it.  As a rule never called.
static __device__ __noinline__ void attend_row(const __nv_bfloat16 *q, const __nv_bfloat16 *K,
                                        const __nv_bfloat16 *V, int n, int c0, float scale,
                                        float ref, float *o) {
  auto lo = [](uint32_t w) { return __uint_as_float(w << 16); };
  auto hi = [](uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); };
  const uint4 *q4 = reinterpret_cast<const uint4 *>(q);
  for (int i = 0; i < n; ++i) {
    const uint4 *k4 = reinterpret_cast<const uint4 *>(K + (size_t)i * 128);
    float s = 0.f;
#pragma unroll 4
    for (int x = 0; x < 16; ++x) {
      const uint4 a = q4[x], b = k4[x];
      s = fmaf(lo(a.x), lo(b.x), fmaf(hi(a.x), hi(b.x), s));
      s = fmaf(lo(a.y), lo(b.y), fmaf(hi(a.y), hi(b.y), s));
      s = fmaf(lo(a.z), lo(b.z), fmaf(hi(a.z), hi(b.z), s));
      s = fmaf(lo(a.w), lo(b.w), fmaf(hi(a.w), hi(b.w), s));
    }
    const float w = ex2(fmaf(s, scale, -ref));
    const uint4 *v4 = reinterpret_cast<const uint4 *>(V + (size_t)i * 128 + c0);
#pragma unroll 1
    for (int x = 0; x < 4; ++x) {
      const uint4 v = v4[x];
      float *p = o + 8 * x;
      p[0] = fmaf(w, lo(v.x), p[0]);
      p[1] = fmaf(w, hi(v.x), p[1]);
      p[2] = fmaf(w, lo(v.y), p[2]);
      p[3] = fmaf(w, hi(v.y), p[3]);
      p[4] = fmaf(w, lo(v.z), p[4]);
      p[5] = fmaf(w, hi(v.z), p[5]);
      p[6] = fmaf(w, lo(v.w), p[6]);
      p[7] = fmaf(w, hi(v.w), p[7]);
    }
  }
}
// NaN where one of v is not finite, else 0.
__device__ __forceinline__ float nonfinite(const float (&v)[32]) {
  const uint64_t zero = pk2(0.f, 0.f);
  uint64_t n[4] = {zero, zero, zero, zero};
#pragma unroll
  for (int x = 0; x < 32; x += 2)
    n[(x >> 1) & 3] = fma2(pk2(v[x], v[x + 1]), zero, n[(x >> 1) & 3]);
  float a, b;
  upk2(add2(add2(n[0], n[1]), add2(n[2], n[3])), a, b);
  return a + b;
}

}  // namespace ptx
}  // namespace kvr
