// Log-sum-exp merge of the partial records of one (new token, query head) by one warp (a7).
// Shared by the combine kernel and by the tensor-core attention kernel's own merge, so that both
// give the same bits: the records are added in slot order, against the maximum of up to 64 of them.
#pragma once

#include "aspd_internal.cuh"

namespace aspd {

template <typename T> __device__ inline T combine_from_f32(float x);
template <> __device__ inline float combine_from_f32<float>(float x) { return x; }
template <> __device__ inline __nv_bfloat16 combine_from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// D / 32 floats of one lane from `at` if u < n; nothing is loaded (the values are undefined) otherwise.
template <int U, int EPL>
__device__ __forceinline__ void ldcg_if_below(float (&x)[EPL], const float* at, int n) {
  if constexpr (EPL == 4)
    asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %5, %6;\n\t@p ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
                 : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]) : "l"(at), "r"(n), "n"(U) : "memory");
  else
    asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %3, %4;\n\t@p ld.global.cg.v2.f32 {%0, %1}, [%2];\n\t}"
                 : "=f"(x[0]), "=f"(x[1]) : "l"(at), "r"(n), "n"(U) : "memory");
}

template <int N, int EPL, int U = 0>
__device__ __forceinline__ void fetch_rows(float (&v)[N][EPL], const float* at, size_t stride, int n) {
  if constexpr (U < N) {
    ldcg_if_below<U>(v[U], at, n);
    fetch_rows<N, EPL, U + 1>(v, at + stride, stride, n);
  }
}

// acc += w * x where w is not 0 (the row of a record that weighs nothing may hold anything)
template <int EPL>
__device__ __forceinline__ void add_row(float (&acc)[EPL], const float (&x)[EPL], float w) {
  if constexpr (EPL == 4)
    asm("{\n\t.reg .pred p;\n\tsetp.neu.f32 p, %8, 0f00000000;\n\t@p fma.rn.f32 %0, %4, %8, %0;\n\t@p fma.rn.f32 %1, %5, %8, %1;\n\t"
        "@p fma.rn.f32 %2, %6, %8, %2;\n\t@p fma.rn.f32 %3, %7, %8, %3;\n\t}"
        : "+f"(acc[0]), "+f"(acc[1]), "+f"(acc[2]), "+f"(acc[3]) : "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(w));
  else
    asm("{\n\t.reg .pred p;\n\tsetp.neu.f32 p, %4, 0f00000000;\n\t@p fma.rn.f32 %0, %2, %4, %0;\n\t@p fma.rn.f32 %1, %3, %4, %1;\n\t}"
        : "+f"(acc[0]), "+f"(acc[1]) : "f"(x[0]), "f"(x[1]), "f"(w));
}

// Records p0 .. p0 + n - 1 of KV-head group member g; lane owns D / 32 consecutive output elements.
// The records are read past L1 (ld.global.cg): inside the attention kernel they were written by
// other CTAs of the same launch.
// Up to 64 records share a maximum: their (max, sum) pairs, two to a lane, and the first 8 * NB of their O rows are
// asked for together, the maximum and the weights are made once, and then every row is a broadcast and D / 32
// multiply-adds a lane, so that a row cut into up to 8 * NB parts costs one round trip to L2.  Every NB takes any number of
// records and gives the same bits: a captured launch keeps its instance while updates of its plan change the cuts.
template <typename T, int D, int NB>
__device__ __forceinline__ void combine_row(const float* __restrict__ ws_o, const float2* __restrict__ ws_ml, int p0, int n, int G,
                                            int g, int lane, T* __restrict__ dst) {
  constexpr int EPL = D / 32, kGroup = 64, kRows = 8 * NB;
  static_assert(kRows <= 32, "a lane holds the weight of one of them");
  float M = -INFINITY, L = 0.f, acc[EPL];
#pragma unroll
  for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
  const float* row = ws_o + ((size_t)p0 * G + g) * D + lane * EPL;
  const float2* pair = ws_ml + (size_t)(p0 + lane) * G + g;
  const size_t stride = (size_t)G * D;
#pragma unroll 1
  for (int g0 = 0; g0 < n; g0 += kGroup, pair += (size_t)kGroup * G) {
    const int cnt = min(kGroup, n - g0);
    float2 ml0 = make_float2(-INFINITY, 0.f), ml1 = ml0;
    if (lane < cnt) ml0 = __ldcg(pair);
    if (lane + 32 < cnt) ml1 = __ldcg(pair + 32 * G);
    float w0 = 0.f, w1 = 0.f;
#pragma unroll 1
    for (int b0 = 0; b0 < cnt; b0 += kRows) {
      float v[kRows][EPL];
      fetch_rows<kRows, EPL>(v, row, stride, cnt - b0);
      row += (kGroup % kRows ? min(kRows, cnt - b0) : kRows) * stride;
      asm volatile("" : "+r"(b0));                 // (one copy of the loop's body, not one for its first turn)
      if (b0 == 0) {
        // records of chunks with no visible key have sum 0
        float mb = fmaxf(ml0.y > 0.f ? ml0.x : -INFINITY, ml1.y > 0.f ? ml1.x : -INFINITY);
#pragma unroll
        for (int o = 16; o; o >>= 1) mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
        const float m_new = fmaxf(M, mb);
        const float alpha = m_new == -INFINITY ? 1.f : exp2f(M - m_new);   // M = -inf: alpha = 0
        M = m_new;
        w0 = ml0.y > 0.f ? exp2f(ml0.x - M) : 0.f;
        w1 = ml1.y > 0.f ? exp2f(ml1.x - M) : 0.f;
        float lw = fmaf(ml0.y, w0, ml1.y * w1);
#pragma unroll
        for (int o = 16; o; o >>= 1) lw += __shfl_xor_sync(0xffffffffu, lw, o);
        L = L * alpha + lw;
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[e] *= alpha;
      }
      float wb = __shfl_sync(0xffffffffu, lane >= b0 ? w0 : w1, b0 + lane);           // of record b0 + lane (the source lane is taken modulo 32)
      if (kGroup % kRows && b0 + lane >= cnt) wb = 0.f;                               // 24 rows: the group's last turn has 16 of them
#pragma unroll
      for (int k = 0; k < kRows; ++k) add_row<EPL>(acc, v[k], __shfl_sync(0xffffffffu, wb, k));
    }
  }
  const float inv = __frcp_rn(L);
#pragma unroll
  for (int e = 0; e < EPL; ++e) dst[lane * EPL + e] = combine_from_f32<T>(acc[e] * inv);
}

}  // namespace aspd
