// Merging a row's partial softmax sums over disjoint sets of keys: with
// m* = max m_t, l* = sum l_t 2^(m_t - m*) and O = sum O_t 2^(m_t - m*) / l*.
// Plain C++ apart from the qualifiers, so the arithmetic is also checked on the host.
#pragma once
#include <cmath>

#include <cuda_runtime.h>

// What a part that gave up (a wait that ran out) leaves as its (m, l): no sum of exponentials is negative.
#define FC_NO_PART make_float2(0.f, -1.f)

template <int COLS>
struct FcRowMerge {
  float m, l, acc[COLS];
  bool whole;  // every part has a result

  __host__ __device__ __forceinline__ FcRowMerge() : m(-INFINITY), l(0.f), whole(true) {
#pragma unroll
    for (int u = 0; u < COLS; ++u) acc[u] = 0.f;
  }

  // The next n <= N parts: their (m, l), with m = -inf past n, and COLS columns of their O.  The reference
  // maximum moves from round to round.
  template <int N>
  __host__ __device__ __forceinline__ void round(const float2 (&ml)[N], const float4 (&o)[N][COLS / 4], int n, bool first) {
    float m_new = m;
#pragma unroll
    for (int q = 0; q < N; ++q) m_new = fmaxf(m_new, ml[q].x);
    // parts whose keys all score -inf for this row have m = -inf, l = 0 and O = 0: a reference of 0 keeps their weights 0
    const float m_use = m_new == -INFINITY ? 0.f : m_new;
    if (!first) {
      const float w = exp2f(m - m_use);
      l *= w;
#pragma unroll
      for (int u = 0; u < COLS; ++u) acc[u] *= w;
    }
    m = m_new;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      if (q >= n) break;
      const float w = exp2f(ml[q].x - m_use);
      whole = whole && !(ml[q].y < 0.f);
      l += ml[q].y * w;
#pragma unroll
      for (int u = 0; u < COLS / 4; ++u) {
        acc[4 * u] += o[q][u].x * w;
        acc[4 * u + 1] += o[q][u].y * w;
        acc[4 * u + 2] += o[q][u].z * w;
        acc[4 * u + 3] += o[q][u].w * w;
      }
    }
  }
};
