// slot_terms.cuh — four genes of one slot, for kernels where one slot per lane is
// a link of the generation's chain.
#pragma once
#include "objectives.cuh"

namespace de {

// Griewank: accum_gene of the genes j0 .. j0 + 3, each term by the same operations
// and added in the same order, but the four terms side by side and both logarithms
// in place of a branch per gene: one latency of sine and logarithm instead of four.
// us per generation, branches -> this: segment rows NEC N = 300, D = 500 3.17 -> 2.75,
// N = 1000, D = 1000 3.57 -> 3.05; binomial rows N = 300, D = 500 3.23 -> 2.88, N = 600, D
// = 100 2.89 -> 2.70; one cluster N = 50, D = 30 NEC 1.70 -> 1.46, N = 100, D = 50 binomial
// 2.18 -> 2.13, N = 200, D = 30 exponential (bound by the walk) 2.96 -> 3.19.
__device__ __forceinline__ void griewank_slot(Acc& a, const float4& x, int j0, const GenParams& p) {
  const float v[4] = {x.x, x.y, x.z, x.w};
  float t[4], n[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float h = sinf(0.5f * (v[e] * rsqrtf((float)(j0 + e + 1))));
    const float c = fmaf(-2.0f * h, h, 1.0f);
    const float l1 = log1pf(-2.0f * h * h), l2 = logf(fabsf(c));
    t[e] = c > 0.5f ? l1 : l2;
    n[e] = c < 0.0f ? 1.0f : 0.0f;
  }
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (j0 + e < p.D) {
      a.a = fmaf(v[e], v[e], a.a);
      a.b += t[e];
      a.c += n[e];
    }
}

}  // namespace de
